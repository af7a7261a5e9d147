// step_d2q9.cuh -- fused pull-stream + FP central-moment collision of the coupled D2Q9 flow
// (Appendix A) and D2Q9 energy (Appendix B) lattices, one node per thread.
//
// The raw -> central map of Steps 1-2 is done as two sweeps of 3-link lines (x, then y), which
// equals P then F on the tensor-product D2Q9 set; Steps 4-5 are the inverse sweeps.
//
// Deviation form: the kernel carries delta_a = f_a - w_a and gamma_a = g_a - w_a T_o.  Because
// the sweeps are linear, the central moments of f are those of the rest populations w at the
// velocity u, K_ab = W_a(ux) W_b(uy) with W_0 = 1, W_1 = -u, W_2 = 1/3 + u^2, plus the central
// moments D_ab of delta.  The relaxation is rewritten for the deviations D_ab -> T_ab
// (kappa~_ab = K_ab + T_ab) with the O(1) parts of K cancelled analytically, so every quantity
// in the collision is small and keeps the register type's full relative precision.
#pragma once

#include "lattices.cuh"
#include "lbm_common.cuh"

namespace lbm {

template <class R>
using Coeffs2D = Coeffs<R, 9, 9>;

// Which lattices a pull reads.
enum { kFlow = 1, kEnergy = 2, kBoth = 3 };

// Streaming (Eqs. LBMsteps-stream, LBMsteps-streamg) with half-way bounce-back for f, and
// bounce-back (adiabatic) or anti-bounce-back (fixed T) for g at the walls (Sec. 6.1), in
// deviations: the anti-bounce-back g_a = -g~_abar + 2 w_a T_w becomes
// gamma_a = -gamma~_abar + 2 w_a (T_w - T_o).
template <class S, class Idx = size_t, int kPull = kPullDev, int kOf = kBoth>
__device__ __forceinline__ void pull_d2q9(const typename S::T* __restrict__ fin,
                                          const typename S::T* __restrict__ gin, const Geometry& geo,
                                          const NodeWalls<typename S::R>& w, int i, typename S::R T_ref,
                                          typename S::R f[9], typename S::R g[9])
{
    using R = typename S::R;
    static_for<9>([&](auto A) {
        constexpr int a = decltype(A)::value;
        constexpr int o = opp9(a);
        bool out, dir;
        R tw;
        const int s = link_source<e9(a, 0), e9(a, 1), 0>(geo, w, i, &out, &dir, &tw);
        const Idx off = out ? (Idx)o * geo.n + i : (Idx)a * geo.n + s;
        if constexpr ((kOf & kFlow) != 0) f[a] = load_link<S, kPull>(fin, off, R(w9(a)));
        if constexpr ((kOf & kEnergy) != 0) {
            const R gv = load_link<S, kPull>(gin, off, R(w9(a)) * T_ref);
            g[a] = dir ? anti_bounce<S, kPull>(gv, w9(a), tw, T_ref) : gv;
        }
    });
}

// The same pull at a node whose eight neighbours all lie inside the box: no wall and no
// periodic wrap touches any link, so every population comes straight from its upwind node.
template <class S, class Idx = size_t, int kPull = kPullDev, int kOf = kBoth>
__device__ __forceinline__ void pull_d2q9_interior(const typename S::T* __restrict__ fin,
                                                   const typename S::T* __restrict__ gin,
                                                   const Geometry& geo, int i, typename S::R T_ref,
                                                   typename S::R f[9], typename S::R g[9])
{
    using R = typename S::R;
    static_for<9>([&](auto A) {
        constexpr int a = decltype(A)::value;
        const Idx off = (Idx)a * geo.n + (i - (e9(a, 0) + e9(a, 1) * geo.nx));
        if constexpr ((kOf & kFlow) != 0) f[a] = load_link<S, kPull>(fin, off, R(w9(a)));
        if constexpr ((kOf & kEnergy) != 0) g[a] = load_link<S, kPull>(gin, off, R(w9(a)) * T_ref);
    });
}

// Flow collision (App. A Step 3; second-order sources vanish; sigma_12 carries the factor 2 of
// Eq. forcing:2D) on the deviations: D[b][a] = kappa_ab - K_ab on entry, kappa~_ab - K_ab on exit.
template <class R>
__device__ __forceinline__ void relax_f_d2q9(R D[3][3], R drho, R irho, R ux, R uy, R Fx, R Fy,
                                             const Coeffs2D<R>& c)
{
    const R third = R(1.0 / 3.0);
    const R A = third + ux * ux, B = third + uy * uy;     // K_20, K_02
    const R uxuy = ux * uy;                                // K_11
    const R D00 = D[0][0], D10 = D[0][1], D20 = D[0][2];
    const R D01 = D[1][0], D11 = D[1][1], D21 = D[1][2];
    const R D02 = D[2][0], D12 = D[2][1], D22 = D[2][2];
    const R Fxr = Fx * irho, Fyr = Fy * irho;
    // sources with the full pre-collision moments kappa = K + D
    const R k11 = uxuy + D11, k20 = A + D20, k02 = B + D02;
    const R k21 = D21 - A * uy, k12 = D12 - ux * B;
    const R s21 = R(2) * Fxr * k11 + Fyr * k20;
    const R s12 = Fxr * k02 + R(2) * Fyr * k11;
    const R s22 = R(2) * (Fxr * k12 + Fyr * k21);

    const R T00 = D00 + c.om_f[0] * (drho - D00);
    const R T10 = D10 - c.om_f[1] * (D10 - ux) + c.hf[1] * Fx;
    const R T01 = D01 - c.om_f[2] * (D01 - uy) + c.hf[2] * Fy;
    const R D2s = D20 + D02, D2d = D20 - D02;
    const R u2s = ux * ux + uy * uy, u2d = ux * ux - uy * uy;
    const R T2s = D2s + c.om_f[3] * (R(2.0 / 3.0) * drho - u2s - D2s);
    const R T2d = D2d - c.om_f[4] * (D2d + u2d);
    const R T11 = D11 - c.om_f[5] * (D11 + uxuy);
    const R T21 = D21 - c.om_f[6] * (D21 - A * uy) + c.hf[6] * s21;
    const R T12 = D12 - c.om_f[7] * (D12 - ux * B) + c.hf[7] * s12;
    const R T20 = R(0.5) * (T2s + T2d);
    const R T02 = R(0.5) * (T2s - T2d);
    // kappa^Mv_22 - K_22 with t20 = A + T20, t02 = B + T02, t11 = uxuy + T11
    const R t11 = uxuy + T11;
    const R M22 = (A * T02 + B * T20 + T20 * T02 + R(2) * t11 * t11 - A * B * drho) * irho;
    const R T22 = D22 + c.om_f[8] * (M22 - D22) + c.hf[8] * s22;

    D[0][0] = T00; D[0][1] = T10; D[0][2] = T20;
    D[1][0] = T01; D[1][1] = T11; D[1][2] = T21;
    D[2][0] = T02; D[2][1] = T12; D[2][2] = T22;
}

// Energy collision in central-moment space on full values (App. B Step 3); n[b][a] holds eta_ab
// on entry and eta~_ab on exit.  The attractors of orders 3-4 come from the post-collision lower
// moments: option A (Eq. MvT2D, c.gopt = 0) or the renormalized option B (Eq. MvT2DoptionB).
template <class R>
__device__ __forceinline__ void relax_g_d2q9(R n[3][3], R T, const Coeffs2D<R>& c)
{
    const R n00 = n[0][0], n10 = n[0][1], n20 = n[0][2];
    const R n01 = n[1][0], n11 = n[1][1], n21 = n[1][2];
    const R n02 = n[2][0], n12 = n[2][1], n22 = n[2][2];
    constexpr double cs2 = 1.0 / 3.0;

    const R t00 = n00 + c.om_g[0] * (T - n00);
    const R t10 = n10 - c.om_g[1] * n10;
    const R t01 = n01 - c.om_g[2] * n01;
    const R n2s = n20 + n02, n2d = n20 - n02;
    const R t2s = n2s + c.om_g[3] * (R(2 * cs2) * T - n2s);
    const R t2d = n2d - c.om_g[4] * n2d;
    const R t11 = n11 - c.om_g[5] * n11;
    const R t20 = R(0.5) * (t2s + t2d);
    const R t02 = R(0.5) * (t2s - t2d);
    R Mv21, Mv12, Mv22;
    if (c.gopt == 0) {
        Mv21 = R(2.0 / 3.0 * cs2) * t01;
        Mv12 = R(2.0 / 3.0 * cs2) * t10;
        Mv22 = R(0.5 * cs2) * (t20 + t02);
    } else {
        const R iT = R(1) / T;
        const R c23 = R(2.0 / 3.0) * iT;
        Mv21 = c23 * (t20 * t01 + R(2) * t11 * t10);
        Mv12 = c23 * (t02 * t10 + R(2) * t11 * t01);
        Mv22 = iT * (t20 * t02 + R(2) * t11 * t11);
    }
    const R t21 = n21 + c.om_g[6] * (Mv21 - n21);
    const R t12 = n12 + c.om_g[7] * (Mv12 - n12);
    const R t22 = n22 + c.om_g[8] * (Mv22 - n22);

    n[0][0] = t00; n[0][1] = t10; n[0][2] = t20;
    n[1][0] = t01; n[1][1] = t11; n[1][2] = t21;
    n[2][0] = t02; n[2][1] = t12; n[2][2] = t22;
}

// Populations (paper order) <-> p[ey+1][ex+1], then the x and y line sweeps.
template <class R>
__device__ __forceinline__ void to_central_d2q9(const R f[9], R p[3][3], R ux, R uy)
{
    static_for<9>([&](auto A) {
        constexpr int a = decltype(A)::value;
        p[e9(a, 1) + 1][e9(a, 0) + 1] = f[a];
    });
#pragma unroll
    for (int j = 0; j < 3; ++j) central_line(p[j][0], p[j][1], p[j][2], ux);
#pragma unroll
    for (int a = 0; a < 3; ++a) central_line(p[0][a], p[1][a], p[2][a], uy);
}

template <class R>
__device__ __forceinline__ void from_central_d2q9(R p[3][3], R f[9], R ux, R uy)
{
#pragma unroll
    for (int a = 0; a < 3; ++a) uncentral_line(p[0][a], p[1][a], p[2][a], uy);
#pragma unroll
    for (int j = 0; j < 3; ++j) uncentral_line(p[j][0], p[j][1], p[j][2], ux);
    static_for<9>([&](auto A) {
        constexpr int a = decltype(A)::value;
        f[a] = p[e9(a, 1) + 1][e9(a, 0) + 1];
    });
}

// Both collisions and the store of one node at the rates lbm_create sets, option A and gravity along
// y (unit_rates_2d, checked by the host), from the stored numbers in f and g (raw).  Used for FP64
// storage, bound by the FP64 pipe, and FP16 storage, bound by issue; FP32 storage, bound by the
// memory, keeps the general collision and with it its rounding.
//
// A moment relaxed at rate 1 lands on its attractor plus half its source, so the collision needs, of the
// flow, rho, j, the two shear moments and the few moments that the force multiplies, and, of the
// energy, T and the first-order moments: they are taken from raw sums of the links, shifted with
// rho u = j + F / 2 (j_x = rho u_x without a force along x).  The relaxed central moments of the flow are held
// as deviations e from the rest state moving at u (1, 1/3 on 20 and 02, 1/9 on 22, times kUnits), whose
// share of the inverse sweeps is the rest weights; so, as in the general form, no O(1) number is rounded
// on the way to the stored one.  The energy's are deviations from T_o times these in FP16 storage and full
// values in FP64 storage, which sums and writes its energy populations as stored (energy_sums_d2q9).
template <class R>
struct FlowSums2D {
    R drho, jx, jy, Mxx, Myy, Mxy, Mxxy;
};
template <class R>
struct EnergySums2D {
    R dT, T, jgx, jgy;
};
// rho and u of a node, and what both collisions share of the force along y (py = rho u_y).
template <class R>
struct Macro2D {
    R rho, irho, Fy, hF, py, ux, uy;
};

template <class S>
__device__ __forceinline__ FlowSums2D<typename S::R> flow_sums_d2q9(const typename S::R f[9])
{
    using R = typename S::R;
    // raw sums of the flow, rows e_y = -1, 0, 1: (7, 4, 8), (3, 0, 1), (6, 2, 5).  For stored
    // populations the rest weights come off exactly: (a - 2 w) + c has no rounding.
    R k0[3], d[3], s[3];
    {
        constexpr int row[3][3] = {{7, 4, 8}, {3, 0, 1}, {6, 2, 5}};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const R a = f[row[j][0]], b = f[row[j][1]], cc = f[row[j][2]];
            d[j] = cc - a;
            if constexpr (S::kFull) {
                s[j] = (a - R(2.0 * w9(row[j][0]))) + cc;
                k0[j] = s[j] + (b - R(w9(row[j][1])));
            } else {
                s[j] = a + cc;
                k0[j] = s[j] + b;
            }
        }
    }
    FlowSums2D<R> m;
    m.Myy = k0[0] + k0[2];
    m.drho = m.Myy + k0[1];
    m.jx = (d[0] + d[2]) + d[1];
    m.jy = k0[2] - k0[0];
    m.Mxx = (s[0] + s[2]) + s[1];
    m.Mxy = d[2] - d[0];
    m.Mxxy = s[2] - s[0];
    return m;
}

// Raw sums of the energy, over opposite links: g = dT + T0.  Stored populations are summed as they are
// (T0 = 0), which also keeps the small ones beside a cold wall exact.  Against 128 bits, T in [0, 1], an update's
// rounding is 1.62e-17 rms on a population and 5.0e-17 on their sum, that of the general collision (full
// moments between rounded rest weights taken off and put on) 1.66e-17 and 5.4e-17 with a drift of the
// sum of 2.8e-17 per update.
template <class S>
__device__ __forceinline__ EnergySums2D<typename S::R> energy_sums_d2q9(const typename S::R g[9],
                                                                        const UnitCoeffs<typename S::R>& c)
{
    using R = typename S::R;
    EnergySums2D<R> m;
    m.dT = (g[0] + ((g[1] + g[3]) + (g[2] + g[4]))) + ((g[5] + g[7]) + (g[6] + g[8]));
    const R d57 = g[5] - g[7], d68 = g[6] - g[8];
    m.jgx = (g[1] - g[3]) + (d57 - d68);
    m.jgy = (g[2] - g[4]) + (d57 + d68);
    m.T = S::kFull ? m.dT : R(S::kUnits) * c.T_ref + m.dT;
    return m;
}

template <class S>
__device__ __forceinline__ Macro2D<typename S::R> macro_d2q9(typename S::R drho, typename S::R jx, typename S::R jy,
                                                             typename S::R dT, const UnitCoeffs<typename S::R>& c)
{
    using R = typename S::R;
    Macro2D<R> m;
    m.rho = R(S::kUnits) + drho;
    m.irho = recip(m.rho);
    m.Fy = c.gbeta * (S::kFull ? dT - c.T_ref : dT);
    m.hF = R(0.5) * m.Fy;
    m.py = jy + m.hF;
    m.ux = jx * m.irho;
    m.uy = m.py * m.irho;
    return m;
}

template <class S>
__device__ __forceinline__ void collide_flow_d2q9_unit(const FlowSums2D<typename S::R>& m, const Macro2D<typename S::R>& u,
                                                       const UnitCoeffs<typename S::R>& c, typename S::R df[9])
{
    using R = typename S::R;
    constexpr double kS = S::kUnits;
    const R third = R(1.0 / 3.0), half = R(0.5);
    const R drho = m.drho, jx = m.jx, Mxx = m.Mxx, Myy = m.Myy, Mxy = m.Mxy, Mxxy = m.Mxxy;
    const R rho = u.rho, irho = u.irho, Fy = u.Fy, hF = u.hF, py = u.py, ux = u.ux, uy = u.uy;
    const R uxh = half * ux, uyh = half * uy;
    R p[3][3];   // [y link][x moment]: x moments of order 1, 2 halved
    {
        // pre-collision central moments of order 2 (e20, e02: less kS / 3) and kappa_21
        const R k11 = (Mxy - jx * uy) + hF * ux;
        const R e20p = Mxx - jx * ux;
        const R e02p = Myy - (py - Fy) * uy;
        const R k20 = R(kS / 3.0) + e20p;
        const R k21 = (Mxxy - uy * k20) - ux * (k11 + Mxy);
        // relaxation and sources (sigma_21 = F_y kappa_20 / rho, sigma_12 = 2 F_y kappa_11 / rho,
        // sigma_22 = 2 F_y kappa_21 / rho), moments of order 1-2 per axis halved per axis
        const R G = Fy * irho;
        const R td = c.kf[0] * (e20p - e02p);
        const R a3 = third * drho;
        const R e20 = a3 + half * td, e02 = a3 - half * td;
        const R t11 = c.kf[1] * k11;
        const R q11 = R(0.25) * t11;
        const R G4 = R(0.25) * G;
        const R q12 = G4 * k11;
        const R h21 = G4 * k20;                 // t21 / 2 = G k20 / 4
        const R e22 = (R(kS / 9.0) * drho + e20 * e02 + (t11 + t11) * t11) * irho + G * k21;
        // y sweep; x moment 0: (kS + drho, F/2, kS/3 + e02)
        {
            const R h1 = half * hF, r1 = half * (py + hF);
            const R r2 = half * e02 + uy * (h1 + r1);
            p[0][0] = r2 - r1;
            p[1][0] = fma_(R(-2), r2, drho);
            p[2][0] = r2 + r1;
        }
        unline0(q11, q12, uy + uy, p[0][1], p[1][1], p[2][1]);
        {   // x moment 2, halved: (kS/6 + e20/2, t21/2, kS/18 + e22/2), orders 1-2 in y halved again
            const R e20h = half * e20;
            unline(e20h, R(kS / 6.0) + e20h, half * h21, R(0.25) * e22, uy, uyh, p[0][2], p[1][2], p[2][2]);
        }
    }
    unline(p[0][0], R(kS / 6.0) + p[0][0], p[0][1], p[0][2], ux, uxh, df[7], df[4], df[8]);
    unline(p[1][0], R(kS * 2.0 / 3.0) + p[1][0], p[1][1], p[1][2], ux, uxh, df[3], df[0], df[1]);
    unline(p[2][0], R(kS / 6.0) + p[2][0], p[2][1], p[2][2], ux, uxh, df[6], df[2], df[5]);

}

template <class S>
__device__ __forceinline__ void collide_energy_d2q9_unit(const EnergySums2D<typename S::R>& m, typename S::R ux,
                                                         typename S::R uy, const UnitCoeffs<typename S::R>& c,
                                                         typename S::R dg[9])
{
    using R = typename S::R;
    const R half = R(0.5), uxh = half * ux, uyh = half * uy;
    const R dT = m.dT, T = m.T, jgx = m.jgx, jgy = m.jgy;
    R p[3][3];
    // energy: T, (1 - omega) eta_1, then c_s^2 T, (2/3) c_s^2 t_1 and c_s^4 T
    {
        const R t10 = c.kg[0] * (jgx - ux * T);
        const R t01 = c.kg[1] * (jgy - uy * T);
        const R dT6 = R(1.0 / 6.0) * dT, T6 = S::kFull ? dT6 : R(1.0 / 6.0) * T;
        unline(dT, T, half * t01, dT6, uy, uyh, p[0][0], p[1][0], p[2][0]);
        {   // x moment 1, halved: (t10, 0, (2/9) t10) / 2
            const R h = half * t10;
            const R r1 = uyh * h, r2 = R(1.0 / 9.0) * h + uy * r1;
            p[0][1] = r2 - r1;
            p[1][1] = fma_(R(-2), r2, h);
            p[2][1] = r2 + r1;
        }
        unline(dT6, T6, R(1.0 / 18.0) * t01, R(1.0 / 36.0) * dT, uy, uyh, p[0][2], p[1][2], p[2][2]);
        if constexpr (S::kFull) {
            unline(p[0][0], p[0][0], p[0][1], p[0][2], ux, uxh, dg[7], dg[4], dg[8]);
            unline(p[1][0], p[1][0], p[1][1], p[1][2], ux, uxh, dg[3], dg[0], dg[1]);
            unline(p[2][0], p[2][0], p[2][1], p[2][2], ux, uxh, dg[6], dg[2], dg[5]);
        } else {
            const R T0 = R(S::kUnits) * c.T_ref;
            const R c6 = R(1.0 / 6.0) * T0, c23 = R(2.0 / 3.0) * T0;
            unline(p[0][0], c6 + p[0][0], p[0][1], p[0][2], ux, uxh, dg[7], dg[4], dg[8]);
            unline(p[1][0], c23 + p[1][0], p[1][1], p[1][2], ux, uxh, dg[3], dg[0], dg[1]);
            unline(p[2][0], c6 + p[2][0], p[2][1], p[2][2], ux, uxh, dg[6], dg[2], dg[5]);
        }
    }

}

template <class S, class Idx>
__device__ __forceinline__ void collide_store_d2q9_unit(const typename S::R f[9], const typename S::R g[9],
                                                        typename S::T* __restrict__ fout,
                                                        typename S::T* __restrict__ gout,
                                                        const Geometry& geo,
                                                        const UnitCoeffs<typename S::R>& c,
                                                        unsigned* status, int i)
{
    using R = typename S::R;
    const FlowSums2D<R> mf = flow_sums_d2q9<S>(f);
    const EnergySums2D<R> mg = energy_sums_d2q9<S>(g, c);
    const Macro2D<R> u = macro_d2q9<S>(mf.drho, mf.jx, mf.jy, mg.dT, c);
    check_node_bits(status, u.rho, mg.T);
    R df[9], dg[9];
    collide_flow_d2q9_unit<S>(mf, u, c, df);
    collide_energy_d2q9_unit<S>(mg, u.ux, u.uy, c, dg);
    if constexpr (std::is_same<S, StoreF16S>::value) {
        store_node_f16s<9, 9, Idx, true>(fout, gout, (Idx)geo.n, i, df, dg, c.fp16_sr);
    } else {
        static_for<9>([&](auto A) {
            constexpr int a = decltype(A)::value;
            S::store_dev(fout, (Idx)a * geo.n + i, df[a], R(w9(a)));
            gout[(Idx)a * geo.n + i] = dg[a];
        });
    }
}

// Macroscopic fields, both collisions and the store of one node at any rates, from the pulled deviations.
template <class S, class Idx>
__device__ __forceinline__ void collide_store_d2q9(typename S::R f[9], typename S::R g[9],
                                                   typename S::T* __restrict__ fout,
                                                   typename S::T* __restrict__ gout, const Geometry& geo,
                                                   const Coeffs2D<typename S::R>& c, unsigned* status, int i)
{
    using R = typename S::R;
    // rho = 1 + sum delta, rho u = sum delta e + F/2, T = T_o + sum gamma (sum w = 1, sum w e = 0)
    const R dT = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];
    const R drho = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
    const R jx = (f[1] + f[5] + f[8]) - (f[3] + f[6] + f[7]);
    const R jy = (f[2] + f[5] + f[6]) - (f[4] + f[7] + f[8]);
    const R Fb = c.gbeta * dT;
    const R Fx = c.gaxis == 0 ? Fb : R(0);
    const R Fy = c.gaxis == 1 ? Fb : R(0);
    const R rho = R(1) + drho;
    const R T = c.T_ref + dT;
    const R irho = R(1) / rho;
    const R ux = (jx + R(0.5) * Fx) * irho;
    const R uy = (jy + R(0.5) * Fy) * irho;
    check_node(status, rho, T);

    R p[3][3];
    to_central_d2q9(f, p, ux, uy);
    relax_f_d2q9(p, drho, irho, ux, uy, Fx, Fy, c);
    from_central_d2q9(p, f, ux, uy);

    // energy populations on full values: g = w T_o + gamma
    static_for<9>([&](auto A) {
        constexpr int a = decltype(A)::value;
        g[a] += R(w9(a)) * c.T_ref;
    });
    to_central_d2q9(g, p, ux, uy);
    relax_g_d2q9(p, T, c);
    from_central_d2q9(p, g, ux, uy);

    if constexpr (std::is_same<S, StoreF16S>::value) {
        if (c.fp16_sr) {
            R dg[9];
            static_for<9>([&](auto A) {
                constexpr int a = decltype(A)::value;
                dg[a] = g[a] - R(w9(a)) * c.T_ref;
            });
            store_node_f16s<9, 9, Idx>(fout, gout, (Idx)geo.n, i, f, dg, 1);
            return;
        }
    }
    static_for<9>([&](auto A) {
        constexpr int a = decltype(A)::value;
        S::store_dev(fout, (Idx)a * geo.n + i, f[a], R(w9(a)));
        S::store_dev(gout, (Idx)a * geo.n + i, g[a] - R(w9(a)) * c.T_ref, R(w9(a)) * c.T_ref);
    });
}

template <class S, bool kUnit>
using StepCoeffs2D = typename std::conditional<kUnit, UnitCoeffs<typename S::R>, Coeffs2D<typename S::R>>::type;

// The pull of one node of the step.
template <class S, class Idx, int kPull, int kOf, class C>
__device__ __forceinline__ void pull_by_warp_d2q9(const typename S::T* __restrict__ fin,
                                                  const typename S::T* __restrict__ gin, const Geometry& geo,
                                                  const C& c, int x, int y, int i, typename S::R f[9],
                                                  typename S::R g[9])
{
    using R = typename S::R;
    // Which pull: decided per warp where possible, so that a warp holding an x-wall node of an
    // interior row runs one x-only pull instead of both the interior and the general pull.
    const bool y_in = y > 0 && y < geo.ny - 1;
    const bool in = y_in && x > 0 && x < geo.nx - 1;
    const unsigned lanes = __activemask();
    if (__all_sync(lanes, in)) {
        pull_d2q9_interior<S, Idx, kPull, kOf>(fin, gin, geo, i, c.T_ref, f, g);
    } else if (__all_sync(lanes, y_in)) {
        const NodeWalls<R> w = node_walls_x<R>(geo, x, y, 0);
        pull_d2q9<S, Idx, kPull, kOf>(fin, gin, geo, w, i, c.T_ref, f, g);
    } else if (in) {
        pull_d2q9_interior<S, Idx, kPull, kOf>(fin, gin, geo, i, c.T_ref, f, g);
    } else {
        const NodeWalls<R> w = node_walls<R>(geo, x, y, 0, 2);
        pull_d2q9<S, Idx, kPull, kOf>(fin, gin, geo, w, i, c.T_ref, f, g);
    }
}

// One time step at one node: pull, macroscopic fields (App. A Step 7, App. B Step 7, Sec. 6.1
// Boussinesq force), collide f and g, store.  kUnit: the reduced collision above.
template <class S, class Idx, bool kUnit = false>
__device__ __forceinline__ void node_step_d2q9(const typename S::T* __restrict__ fin,
                                               const typename S::T* __restrict__ gin,
                                               typename S::T* __restrict__ fout,
                                               typename S::T* __restrict__ gout, const Geometry& geo,
                                               const StepCoeffs2D<S, kUnit>& c, unsigned* status,
                                               int x, int y)
{
    using R = typename S::R;
    constexpr int kPull = kPullAfter | (kUnit ? kPullRaw : kPullDev);
    const int i = x + geo.nx * y;
    R f[9], g[9];
    pull_by_warp_d2q9<S, Idx, kPull, kBoth>(fin, gin, geo, c, x, y, i, f, g);
    if constexpr (kUnit) {
        collide_store_d2q9_unit<S, Idx>(f, g, fout, gout, geo, c, status, i);
    } else {
        collide_store_d2q9<S, Idx>(f, g, fout, gout, geo, c, status, i);
    }
}

template <class S, class Idx, bool kUnit = false>
__global__ void __launch_bounds__(256)
    step_d2q9_kernel(const typename S::T* __restrict__ fin, const typename S::T* __restrict__ gin,
                     typename S::T* __restrict__ fout, typename S::T* __restrict__ gout, Geometry geo,
                     StepCoeffs2D<S, kUnit> c, unsigned* status, bool flip)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = (flip ? gridDim.y - 1 - blockIdx.y : blockIdx.y) * blockDim.y + threadIdx.y;
    wait_previous_step();
    if (x >= geo.nx || y >= geo.ny) return;
    node_step_d2q9<S, Idx, kUnit>(fin, gin, fout, gout, geo, c, status, x, y);
}

// FP16 storage, reduced collision, two x-adjacent nodes per thread (x even); see
// step_d3q27_pair_f16s_kernel.  A node takes 15 loads and 9 stores instead of 18 and 18.
// 4096 x 2048: 105 us per step against 133 (issue slots 73 % busy at 2048^2, ncu); 1024 x 512, in L2, 7.9 against 8.5; 512^2 is even, and smaller
// boxes lose warps.  Bitwise the results of the one-node kernel.
__device__ __forceinline__ void pair_node_d2q9(const float f[9], const float g[9], const UnitCoeffs<float>& c,
                                               unsigned* status, int i, unsigned h2[9])
{
    using S = StoreF16S;
    const FlowSums2D<float> mf = flow_sums_d2q9<S>(f);
    const EnergySums2D<float> mg = energy_sums_d2q9<S>(g, c);
    const Macro2D<float> u = macro_d2q9<S>(mf.drho, mf.jx, mf.jy, mg.dT, c);
    check_node_bits(status, u.rho, mg.T);
    float df[9], dg[9];
    collide_flow_d2q9_unit<S>(mf, u, c, df);
    collide_energy_d2q9_unit<S>(mg, u.ux, u.uy, c, dg);
    if (c.fp16_sr) pack_node_f16s<9, 9, true, true>(i, df, dg, h2);
    else pack_node_f16s<9, 9, false, true>(i, df, dg, h2);
}

// The values of a node on an x wall (or x wrap) of an interior row that arrive through x.
__device__ __forceinline__ void fix_x_edge_d2q9_f16s(const __half* __restrict__ fin, const __half* __restrict__ gin,
                                                     const Geometry& geo, int x, int y, int i, float T_ref, float f[9],
                                                     float g[9])
{
    using S = StoreF16S;
    const NodeWalls<float> w = node_walls_x<float>(geo, x, y, 0);
    static_for<9>([&](auto A) {
        constexpr int a = decltype(A)::value;
        constexpr int ex = e9(a, 0), o = opp9(a);
        if constexpr (ex != 0) {
            if (ex == 1 ? x == 0 : x == geo.nx - 1) {
                bool out, dir;
                float tw;
                const int s = link_source<ex, e9(a, 1), 0>(geo, w, i, &out, &dir, &tw);
                const unsigned off = out ? (unsigned)o * geo.n + i : (unsigned)a * geo.n + s;
                f[a] = S::raw(ld_step(fin + off));
                const float gv = S::raw(ld_step(gin + off));
                g[a] = dir ? anti_bounce<S, kPullRaw>(gv, w9(a), tw, T_ref) : gv;
            }
        }
    });
}

template <class Idx>
__global__ void __launch_bounds__(256)
    step_d2q9_pair_f16s_kernel(const __half* __restrict__ fin, const __half* __restrict__ gin, __half* __restrict__ fout,
                               __half* __restrict__ gout, Geometry geo, UnitCoeffs<float> c, unsigned* status, bool flip)
{
    using S = StoreF16S;
    const int x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = (flip ? gridDim.y - 1 - blockIdx.y : blockIdx.y) * blockDim.y + threadIdx.y;
    wait_previous_step();
    if (x >= geo.nx || y >= geo.ny) return;
    const int i = x + geo.nx * y;
    const Idx n = (Idx)geo.n;
    unsigned out0[9], out1[9];
    float f[9], g[9];
    if (y > 0 && y < geo.ny - 1) {
        unsigned w[18];
        // an x link that would leave the row reads its partner's place instead and is replaced below: the
        // row behind the last one may end the buffer
        const int lo = x > 0 ? i - 1 : i, hi = x + 2 < geo.nx ? i + 2 : i + 1;
        static_for<18>([&](auto A) {
            constexpr int k = decltype(A)::value, a = k % 9, ex = e9(a, 0);
            const __half* p = (k < 9 ? fin : gin) + (Idx)a * n;
            const int row = e9(a, 1) * geo.nx;
            if constexpr (ex == 0) {
                w[k] = ld_step_pair(p + (i - row));
            } else {
                const int s0 = (ex == 1 ? lo : i + 1) - row, s1 = (ex == 1 ? i : hi) - row;
                w[k] = (unsigned)__half_as_ushort(ld_step(p + s0)) | (unsigned)__half_as_ushort(ld_step(p + s1)) << 16;
            }
        });
        static_for<9>([&](auto A) {
            constexpr int a = decltype(A)::value;
            f[a] = S::raw(low_half(w[a]));
            g[a] = S::raw(low_half(w[9 + a]));
        });
        if (x == 0) fix_x_edge_d2q9_f16s(fin, gin, geo, x, y, i, c.T_ref, f, g);
        pair_node_d2q9(f, g, c, status, i, out0);
        static_for<9>([&](auto A) {
            constexpr int a = decltype(A)::value;
            f[a] = S::raw(high_half(w[a]));
            g[a] = S::raw(high_half(w[9 + a]));
        });
        if (x + 2 == geo.nx) fix_x_edge_d2q9_f16s(fin, gin, geo, x + 1, y, i + 1, c.T_ref, f, g);
    } else {
        constexpr int kPull = kPullAfter | kPullRaw;
        pull_d2q9<S, Idx, kPull>(fin, gin, geo, node_walls<float>(geo, x, y, 0, 2), i, c.T_ref, f, g);
        pair_node_d2q9(f, g, c, status, i, out0);
        pull_d2q9<S, Idx, kPull>(fin, gin, geo, node_walls<float>(geo, x + 1, y, 0, 2), i + 1, c.T_ref, f, g);
    }
    pair_node_d2q9(f, g, c, status, i + 1, out1);
    static_for<18>([&](auto A) {
        constexpr int a = decltype(A)::value;
        const unsigned v = __byte_perm(out0[a / 2], out1[a / 2], (a & 1) ? 0x7632 : 0x5410);
        __half* p = (a < 9 ? fout : gout) + (Idx)(a % 9) * n;
        *reinterpret_cast<unsigned*>(p + i) = v;
    });
}

// FP64, reduced collision, small boxes: the two lattices of 32 nodes on two warps of a block, which swap
// their sums (T, and rho and j) once.  A sub-partition takes an FP64 instruction per 64 cycles however
// few lanes or warps it has, so while warps are fewer than the 608 sub-partitions the step lasts as
// long as one warp's FP64 instructions: about 105 here (the flow's) against 175.  64^2: 5.4 us per step
// against 7.6, 96^2 6.0 against 7.6; with more warps than sub-partitions the second macro_d2q9 only
// costs (128^2 8.7 against 8.3).
// Each warp's arithmetic is that of the one-warp kernel; the states are bitwise the same.
template <class Idx>
__global__ void __launch_bounds__(64)
    step_d2q9_split_f64_kernel(const double* __restrict__ fin, const double* __restrict__ gin, double* __restrict__ fout,
                               double* __restrict__ gout, Geometry geo, UnitCoeffs<double> c, unsigned* status)
{
    using S = StoreF64;
    __shared__ double swap[4][32];
    const int lane = threadIdx.x & 31;
    const bool flow = threadIdx.x < 32;
    const int x = blockIdx.x * 32 + lane, y = blockIdx.y;
    const int i = x + geo.nx * y;
    const bool active = x < geo.nx;
    wait_previous_step();
    double v[9], out[9];
    FlowSums2D<double> mf{};
    EnergySums2D<double> mg{};
    if (active) {
        if (flow) {
            pull_by_warp_d2q9<S, Idx, kPullAfter | kPullRaw, kFlow>(fin, gin, geo, c, x, y, i, v, v);
            mf = flow_sums_d2q9<S>(v);
            swap[0][lane] = mf.drho;
            swap[1][lane] = mf.jx;
            swap[2][lane] = mf.jy;
        } else {
            pull_by_warp_d2q9<S, Idx, kPullAfter | kPullRaw, kEnergy>(fin, gin, geo, c, x, y, i, v, v);
            mg = energy_sums_d2q9<S>(v, c);
            swap[3][lane] = mg.dT;
        }
    }
    __syncthreads();
    if (!active) return;
    const Macro2D<double> u = macro_d2q9<S>(swap[0][lane], swap[1][lane], swap[2][lane], swap[3][lane], c);
    if (flow) {
        collide_flow_d2q9_unit<S>(mf, u, c, out);
        static_for<9>([&](auto A) {
            constexpr int a = decltype(A)::value;
            S::store_dev(fout, (Idx)a * geo.n + i, out[a], w9(a));
        });
    } else {
        check_node_bits(status, u.rho, mg.T);
        collide_energy_d2q9_unit<S>(mg, u.ux, u.uy, c, out);
        static_for<9>([&](auto A) {
            constexpr int a = decltype(A)::value;
            gout[(Idx)a * geo.n + i] = out[a];
        });
    }
}

}  // namespace lbm

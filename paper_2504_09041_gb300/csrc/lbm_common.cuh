// lbm_common.cuh -- storage policies, geometry and the pull-with-walls link for the fused
// collide-and-stream kernels of the Fokker-Planck central-moment LBM (arXiv 2504.09041).
//
// Layout in HBM: structure of arrays, one plane per link, f[a * n + i] with the node index
// i = x + nx * (y + ny * z) (x fastest).  Two buffers per lattice (A -> B, then swap): the
// kernels pull from the post-collision state of the previous step and write the new
// post-collision state at the node itself, so every store is fully coalesced.
#pragma once

#include <cuda_fp16.h>
#include <cstdint>
#include <utility>
#include <type_traits>

namespace lbm {

enum FaceKind { kPeriodic = 0, kAdiabatic = 1, kFixedT = 2 };

// 2D steps of one time loop are launched as programmatic dependents (launch_step_kernel): a step's
// blocks may start once those of the step before it have exited, and wait here for it to complete
// before their first access to populations, so at most two steps are ever in flight.  That hides the
// launch (in graphs, 64^2: FP64 5.7 -> 5.4 us, FP32 1.92 -> 1.73; 512^2 FP32 6.0 -> 5.8; in a stream, 64^2 FP32 4.1 ->
// 2.65).  The 3D steps are launched one after the other: their times do not change.
__device__ __forceinline__ void wait_previous_step() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// After the wait: the next step's blocks may start already, beside this one's.  Where a step's blocks take
// more than half of the GPU's places but not all, those of the next one that find none left crowd onto
// the SMs that come free first, and the step lasts as long as a full SM's (2D FP32 372 x 277 4.35 us
// against 3.15 without, 65 x 1000 4.1 against 3.1; FP64 288 x 288 51 against 32); elsewhere the single boxes gain nothing
// from it, and it is left to adjoint steps that fill the GPU and batches that do not fill it in part.
__device__ __forceinline__ void release_next_step()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Loads of populations: ld_ro through the read-only path, ld_step in kernels that call
// wait_previous_step, whose predecessor writes what they read (volatile, so that they stay behind the
// wait, and not the read-only path).  FP32 and FP16 carry an L2 prefetch hint of 256 bytes: the pull
// reads every population plane in full, so the sectors around each warp's row are always used by
// the neighbouring warps.
__device__ __forceinline__ double ld_ro(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ld_ro(const float* p)
{
    float v;
    asm("ld.global.nc.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ __half ld_ro(const __half* p)
{
    unsigned short v;
    asm("ld.global.nc.L2::256B.b16 %0, [%1];" : "=h"(v) : "l"(p));
    return __ushort_as_half(v);
}
// two neighbouring FP16 values; p on 4 bytes
__device__ __forceinline__ unsigned ld_ro_pair(const __half* p)
{
    unsigned v;
    asm("ld.global.nc.L2::256B.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double ld_step(const double* p)
{
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_step(const float* p)
{
    float v;
    asm volatile("ld.global.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ __half ld_step(const __half* p)
{
    unsigned short v;
    asm volatile("ld.global.L2::256B.b16 %0, [%1];" : "=h"(v) : "l"(p));
    return __ushort_as_half(v);
}

// Storage policies: the type in HBM and the type of the moment algebra in registers.  The
// kernels work on deviations from the rest populations (f_a - w_a and g_a - w_a T_o), which keeps
// every quantity of the collision small and resolves it to the register type's precision.
//  - F64 stores the populations themselves and forms the deviation on load.
//  - F32 stores the deviations.
//  - F16S stores the deviations scaled by 2^10, so that deviations down to 6e-8 stay in FP16's
//    normal range (full 11-bit significand) while |deviation| < 64 still fits; the scale is a
//    power of two and adds no rounding.
//
// The reduced steps (default rates and gravity axis; FP64 and F16S) take the stored number itself (raw) and
// work in its units: every relation of the step is homogeneous of degree one in the populations, so
// multiplying them all by kUnits only multiplies the rest state's constants.  kFull: the stored
// number is the population, not its deviation; the rest state is then taken off in the raw sums (of the
// flow and, in 3D, of the energy; in 2D the energy is summed and written as stored, see
// energy_sums_d2q9).
struct StoreF64 {
    using T = double;
    using R = double;
    static constexpr bool kFull = true;
    static constexpr double kUnits = 1.0;
    __device__ static R raw(T v) { return v; }
    __device__ static R dev(T v, R shift) { return v - shift; }
    __device__ static void store_dev(T* p, size_t i, R dev, R shift) { p[i] = shift + dev; }
};
struct StoreF32 {
    using T = float;
    using R = float;
    __device__ static R dev(T v, R) { return v; }
    __device__ static void store_dev(T* p, size_t i, R dev, R) { p[i] = dev; }
};
struct StoreF16S {
    using T = __half;
    using R = float;
    static constexpr int kScaleLog2 = 10;
    static constexpr float kScale = 1024.0f;   // 2^kScaleLog2
    static constexpr float kInvScale = 1.0f / 1024.0f;
    static constexpr bool kFull = false;
    static constexpr double kUnits = 1024.0;
    __device__ static R raw(T v) { return __half2float(v); }
    __device__ static R dev(T v, R) { return __half2float(v) * kInvScale; }
    __device__ static void store_dev(T* p, size_t i, R dev, R) { p[i] = __float2half_rn(dev * kScale); }
    // a deviation already multiplied by kScale
    __device__ static void store_scaled(T* p, size_t i, R scaled) { p[i] = __float2half_rn(scaled); }
    // Two deviations, already multiplied by kScale, converted together with stochastic rounding: each
    // is rounded up or down to a neighbouring FP16 value with probabilities that make the rounding
    // unbiased, driven by the caller's random bits (Blackwell's cvt.rs).  Returns
    // (half of s0) | (half of s1) << 16.
    __device__ static unsigned pack_sr_scaled(R s0, R s1, unsigned rbits)
    {
        unsigned h2;
        asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(h2) : "f"(s1), "f"(s0), "r"(rbits));
        return h2;
    }
};

// 32-bit integer mix (the "lowbias32" constants of C. Wellons' hash prospector): a counter-style
// source of random bits for stochastic rounding.
__device__ __forceinline__ unsigned mix32(unsigned x)
{
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return x;
}

// Seed of the stochastic rounding of node i: one full mix of the node index and the FP32 bits of two
// of the node's new values, so the bits are reproducible and change whenever an update below half
// an FP16 step changes the node's state.
__device__ __forceinline__ unsigned sr_seed(unsigned i, float d0, float d1)
{
    return mix32(i * 0x9e3779b9u + (__float_as_uint(d0) ^ (__float_as_uint(d1) << 7)));
}

// Random bits of value pair k of a node: the seed times a distinct odd constant.  Multiplication by
// an odd constant permutes the 32-bit words, so every bit of every pair's word is uniformly
// distributed when the seed is, which is all that unbiased rounding needs.
template <int K>
__device__ __forceinline__ unsigned sr_pair_bits(unsigned seed)
{
    constexpr unsigned mult = 0x9e3779b9u + 2u * (unsigned)K * 0x632be5abu;  // odd for every K
    return seed * mult;
}


// The storage forms that have reduced steps: FP64, bound by the FP64 pipe, and FP16, bound by issue.
// FP32 storage is bound by the memory and keeps the general collisions with their rounding.
template <class S>
struct has_unit_step : std::integral_constant<bool, !std::is_same<S, StoreF32>::value> {};

// Loads of two neighbouring FP16 values in a kernel that has called wait_previous_step; p on 4 bytes.
__device__ __forceinline__ unsigned ld_step_pair(const __half* p)
{
    unsigned v;
    asm volatile("ld.global.L2::256B.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ __half low_half(unsigned w) { return __ushort_as_half((unsigned short)(w & 0xffffu)); }
__device__ __forceinline__ __half high_half(unsigned w) { return __ushort_as_half((unsigned short)(w >> 16)); }

// Box geometry and wall description shared by every kernel.
struct Geometry {
    int nx, ny, nz;
    int nxy;                  // nx * ny
    int n;                    // nx * ny * nz (< 2^31)
    int kind[6];              // FaceKind of -x, +x, -y, +y, -z, +z
    double T_wall[6];         // uniform wall temperature of fixed-T faces
    const double* profile[6]; // per-node wall temperature (face tangential order) or nullptr
};

// Relaxation rates and coupling in the register type.
template <class R, int QF, int QG>
struct Coeffs {
    R om_f[QF];   // omega of each relaxed flow moment
    R hf[QF];     // 1 - omega/2 (source weight)
    R om_g[QG];
    R gbeta, T_ref;
    int gaxis;    // 0, 1, 2
    int gopt;     // energy attractors of orders 3-4: 0 = option A, 1 = option B (renormalized)
    int fp16_sr;  // F16S storage: 1 = stochastic rounding of the stored deviations, 0 = nearest
};

// What the reduced steps (default rates and gravity axis) take instead, formed once on the host: their
// FP64 pipe is their bound, so no constant is formed per thread.
template <class R>
struct UnitCoeffs {
    R kf[6];             // 1 - omega of flow slots 4 .. 9
    R kg[3];             // 1 - omega of energy slots 1 .. 3
    R gbeta, T_ref;
    R rest_g[3];         // 3D, FP64 storage: rest values w_b T_ref of energy links 0, 1-6 and 7-14 ...
    R rest_T;            // ... and their sum over the 15 links (T_ref in the other forms)
    int fp16_sr;         // as in Coeffs
};

// Per-thread wall bookkeeping for the pull.  For an axis, "m" is a link whose source lies at
// coordinate - 1 (component +1) and "p" one whose source lies at coordinate + 1 (component -1).
template <class R>
struct NodeWalls {
    int wrap_m[3], wrap_p[3];   // linear-index correction when a periodic axis wraps
    bool out_m[3], out_p[3];    // the source lies beyond a wall
    bool fix_m[3], fix_p[3];    // ... and that wall has a fixed temperature
    R tw_m[3], tw_p[3];         // wall temperature of that fixed-T face at this node
};

// Wall temperature of face f seen from node (x, y, z).
__device__ __forceinline__ double wall_temperature(const Geometry& g, int f, int x, int y, int z)
{
    const double* p = g.profile[f];
    if (p == nullptr) return g.T_wall[f];
    const int ax = f >> 1;
    const int t = ax == 0 ? y + g.ny * z : (ax == 1 ? x + g.nx * z : x + g.nx * y);
    return __ldg(p + t);
}

template <class R>
__device__ __forceinline__ NodeWalls<R> node_walls(const Geometry& g, int x, int y, int z, int dims)
{
    NodeWalls<R> w;
    const int c[3] = {x, y, z};
    const int ext[3] = {g.nx, g.ny, g.nz};
    const int stride[3] = {1, g.nx, g.nxy};
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const bool lo = c[ax] == 0, hi = c[ax] == ext[ax] - 1;
        const bool per = ax >= dims || g.kind[2 * ax] == kPeriodic;
        w.wrap_m[ax] = (lo && per) ? ext[ax] * stride[ax] : 0;
        w.wrap_p[ax] = (hi && per) ? -ext[ax] * stride[ax] : 0;
        w.out_m[ax] = lo && !per;
        w.out_p[ax] = hi && !per;
        w.fix_m[ax] = w.out_m[ax] && g.kind[2 * ax] == kFixedT;
        w.fix_p[ax] = w.out_p[ax] && g.kind[2 * ax + 1] == kFixedT;
        w.tw_m[ax] = w.fix_m[ax] ? R(wall_temperature(g, 2 * ax, x, y, z)) : R(0);
        w.tw_p[ax] = w.fix_p[ax] ? R(wall_temperature(g, 2 * ax + 1, x, y, z)) : R(0);
    }
    return w;
}

// The same bookkeeping for a node whose y and z neighbours all lie inside the box: only the x
// axis can wrap or meet a wall, and the y / z entries are compile-time zeros that fold away.
template <class R>
__device__ __forceinline__ NodeWalls<R> node_walls_x(const Geometry& g, int x, int y, int z)
{
    NodeWalls<R> w;
    const bool lo = x == 0, hi = x == g.nx - 1;
    const bool per = g.kind[0] == kPeriodic;
    w.wrap_m[0] = (lo && per) ? g.nx : 0;
    w.wrap_p[0] = (hi && per) ? -g.nx : 0;
    w.out_m[0] = lo && !per;
    w.out_p[0] = hi && !per;
    w.fix_m[0] = w.out_m[0] && g.kind[0] == kFixedT;
    w.fix_p[0] = w.out_p[0] && g.kind[1] == kFixedT;
    w.tw_m[0] = w.fix_m[0] ? R(wall_temperature(g, 0, x, y, z)) : R(0);
    w.tw_p[0] = w.fix_p[0] ? R(wall_temperature(g, 1, x, y, z)) : R(0);
#pragma unroll
    for (int ax = 1; ax < 3; ++ax) {
        w.wrap_m[ax] = w.wrap_p[ax] = 0;
        w.out_m[ax] = w.out_p[ax] = false;
        w.fix_m[ax] = w.fix_p[ax] = false;
        w.tw_m[ax] = w.tw_p[ax] = R(0);
    }
    return w;
}

// Order of the faces for links that cross two or three walls at an edge or corner of the box:
// the crossed face latest in the order -z, -y, -x, +x, +y, +z (the order of the neighbours'
// linear indices) decides the link's rule.  rank(axis, c) of the face that a link with component
// c = +1 (source at coordinate - 1: the - face) or c = -1 (the + face) crosses on that axis.
__host__ __device__ constexpr int face_rank(int ax, int c)
{
    return c == 1 ? 2 - ax : 3 + ax;
}

// Source of the link arriving at node i along (EX, EY, EZ) after the walls.  Returns the
// linear index of the source node.  *out is set when the source lies beyond a wall.  The crossed
// wall that decides the rule is the one of highest face_rank: *dir is set when it has a fixed
// temperature (anti-bounce-back), and *tw is then its temperature; otherwise the link bounces
// back.  Faces crossed by an edge or corner link therefore decide in the order above.
template <int EX, int EY, int EZ, class R>
__device__ __forceinline__ int link_source(const Geometry& g, const NodeWalls<R>& w, int i,
                                           bool* out, bool* dir, R* tw)
{
    int s = i - (EX + EY * g.nx + EZ * g.nxy);
    bool o = false;
    if (EX == 1) { s += w.wrap_m[0]; o |= w.out_m[0]; }
    if (EX == -1) { s += w.wrap_p[0]; o |= w.out_p[0]; }
    if (EY == 1) { s += w.wrap_m[1]; o |= w.out_m[1]; }
    if (EY == -1) { s += w.wrap_p[1]; o |= w.out_p[1]; }
    if (EZ == 1) { s += w.wrap_m[2]; o |= w.out_m[2]; }
    if (EZ == -1) { s += w.wrap_p[2]; o |= w.out_p[2]; }
    // the deciding face: visit the crossed axes from the highest face rank down
    bool decided = false, d = false;
    R t = R(0);
    constexpr int e[3] = {EX, EY, EZ};
#pragma unroll
    for (int r = 5; r >= 0; --r) {
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            if (e[ax] == 0 || face_rank(ax, e[ax]) != r) continue;
            const bool crossed = e[ax] == 1 ? w.out_m[ax] : w.out_p[ax];
            const bool fixed = e[ax] == 1 ? w.fix_m[ax] : w.fix_p[ax];
            if (crossed && !decided) {
                decided = true;
                d = fixed;
                t = e[ax] == 1 ? w.tw_m[ax] : w.tw_p[ax];
            }
        }
    }
    *out = o;
    *dir = d;
    *tw = d ? t : R(0);
    return s;
}

// How a pull reads populations.
enum Pull {
    kPullDev = 0,    // deviations
    kPullRaw = 1,    // stored numbers, for the reduced steps
    kPullAfter = 2   // flag: in a kernel that has called wait_previous_step
};

template <class S, int kPull, class Idx>
__device__ __forceinline__ typename S::R load_link(const typename S::T* p, Idx off, typename S::R shift)
{
    typename S::T v;
    if constexpr ((kPull & kPullAfter) != 0) v = ld_step(p + off);
    else v = ld_ro(p + off);
    if constexpr ((kPull & kPullRaw) != 0) return S::raw(v);
    else return S::dev(v, shift);
}
// Anti-bounce-back of the energy population gv against a wall at temperature tw (link weight w), in
// the units of load_link.
template <class S, int kPull>
__device__ __forceinline__ typename S::R anti_bounce(typename S::R gv, double w, typename S::R tw,
                                                     typename S::R T_ref)
{
    using R = typename S::R;
    if constexpr ((kPull & kPullRaw) != 0) {
        if constexpr (S::kFull) return R(2.0 * w) * tw - gv;
        else return R(2.0 * S::kUnits * w) * (tw - T_ref) - gv;
    } else {
        return R(2.0 * w) * (tw - T_ref) - gv;
    }
}

__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }

// One line of an inverse sweep whose moments of order 1 and 2 come in halved (h1, h2) and whose
// order-0 moment is split into a constant and the rest k0: (k0 + const, 2 h1, 2 h2 + const / 3) at
// velocity u -> the deviations of the three links from the constant's rest weights.  k0f is the full
// order-0 moment and uh = u / 2.  Six operations; the halvings of uncentral_line are carried by the
// inputs instead (exact: powers of two).  The fused operations are written out: from k0 - 2 r2 the
// compiler makes two additions.
template <class R>
__device__ __forceinline__ void unline(R k0, R k0f, R h1, R h2, R u, R uh, R& a, R& b, R& c)
{
    const R r1 = fma_(uh, k0f, h1);          // half the raw first moment
    const R r2 = fma_(u, h1 + r1, h2);       // half the raw second moment (deviation)
    a = r2 - r1;
    b = fma_(R(-2), r2, k0);
    c = r2 + r1;
}
// The same with a zero order-0 moment; u2 = 2 u.
template <class R>
__device__ __forceinline__ void unline0(R h1, R h2, R u2, R& a, R& b, R& c)
{
    const R r2 = fma_(u2, h1, h2);
    a = r2 - h1;
    b = R(-2) * r2;
    c = r2 + h1;
}

// Compile-time loop: calls f(std::integral_constant<int, 0>), ..., f(<N-1>).
template <class F, int... Is>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, Is...>)
{
    (f(std::integral_constant<int, Is>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& f)
{
    static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// One node's q deviations (flow planes then energy planes) rounded to FP16 storage in pairs: word k
// holds values 2k and 2k + 1.  kStochastic: with the node's random bits (see sr_seed); kScaled: df and
// dg are already multiplied by the storage scale (the seed is still taken from the unscaled bits).
template <int QF, int QG, bool kStochastic, bool kScaled>
__device__ __forceinline__ void pack_node_f16s(int i, const float* df, const float* dg, unsigned h2[(QF + QG) / 2])
{
    constexpr int Q = QF + QG;
    static_assert(Q % 2 == 0, "values are converted in pairs");
    const float unscale = kScaled ? StoreF16S::kInvScale : 1.0f, scale = kScaled ? 1.0f : StoreF16S::kScale;
    const unsigned seed = kStochastic ? sr_seed((unsigned)i, df[0] * unscale, dg[0] * unscale) : 0u;
    static_for<Q / 2>([&](auto K) {
        constexpr int k = decltype(K)::value;
        constexpr int a0 = 2 * k, a1 = 2 * k + 1;
        // value a of the node: flow plane a, or energy plane a - QF (indices kept in range)
        constexpr int f0 = a0 < QF ? a0 : 0, g0 = a0 < QF ? 0 : a0 - QF;
        constexpr int f1 = a1 < QF ? a1 : 0, g1 = a1 < QF ? 0 : a1 - QF;
        const float v0 = a0 < QF ? df[f0] : dg[g0];
        const float v1 = a1 < QF ? df[f1] : dg[g1];
        if constexpr (kStochastic) {
            h2[k] = StoreF16S::pack_sr_scaled(v0 * scale, v1 * scale, sr_pair_bits<k>(seed));
        } else {
            const __half2 h = __floats2half2_rn(v0 * scale, v1 * scale);
            h2[k] = *reinterpret_cast<const unsigned*>(&h);
        }
    });
}

// Store of one node's packed values.
template <int QF, int QG, class Idx>
__device__ __forceinline__ void store_packed_f16s(__half* __restrict__ fout, __half* __restrict__ gout, Idx n, int i,
                                                  const unsigned h2[(QF + QG) / 2])
{
    static_for<QF + QG>([&](auto A) {
        constexpr int a = decltype(A)::value;
        const __half h = __ushort_as_half((unsigned short)(a & 1 ? h2[a / 2] >> 16 : h2[a / 2] & 0xffffu));
        if constexpr (a < QF) fout[(Idx)a * n + i] = h;
        else gout[(Idx)(a - QF) * n + i] = h;
    });
}

// Store of one node's deviations through F16S storage; sr: stochastic rounding.
template <int QF, int QG, class Idx, bool kScaled = false>
__device__ __forceinline__ void store_node_f16s(__half* __restrict__ fout, __half* __restrict__ gout, Idx n, int i,
                                                const float* df, const float* dg, int sr)
{
    unsigned h2[(QF + QG) / 2];
    if (sr) {
        pack_node_f16s<QF, QG, true, kScaled>(i, df, dg, h2);
        store_packed_f16s<QF, QG, Idx>(fout, gout, n, i, h2);
    } else {
        pack_node_f16s<QF, QG, false, kScaled>(i, df, dg, h2);
        store_packed_f16s<QF, QG, Idx>(fout, gout, n, i, h2);
    }
}

// 1 / x within an ulp, for x away from the ends of the range (0 and infinity give NaN): the hardware's
// approximation y and a Householder step in its residual e = 1 - x y, which is exact to rounding:
// 1 / x = y (1 + e + e^2 + ...), cubic for double (y has about 20 bits), to order e (Newton's) for
// float.  Three FP64 operations instead of the eight or so of an IEEE division, whose last half ulp the
// velocity does not need.
__device__ __forceinline__ double recip(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ float recip(float x)
{
    float y;
    asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return fmaf(y, fmaf(-x, y, 1.0f), y);
}

// Divergence flag: bit 0 set when a node sees a non-finite or non-positive density or a
// non-finite temperature.
template <class R>
__device__ __forceinline__ void check_node(unsigned* status, R rho, R T)
{
    if (!(rho > R(0)) || !(fabs(T) < R(1e30)) || !(rho < R(1e30))) atomicOr(status, 1u);
}

// The same test of FP64 values on their bits, off the FP64 pipe: 0x46293e59 is the high word of 1e30.
__device__ __forceinline__ void check_node_bits(unsigned* status, double rho, double T)
{
    const int hr = __double2hiint(rho), ht = __double2hiint(T) & 0x7fffffff;
    const bool positive = hr > 0 || (hr == 0 && __double2loint(rho) != 0);
    if (!positive || hr >= 0x46293e59 || ht >= 0x46293e59) atomicOr(status, 1u);
}
__device__ __forceinline__ void check_node_bits(unsigned* status, float rho, float T)
{
    check_node(status, rho, T);
}

}  // namespace lbm

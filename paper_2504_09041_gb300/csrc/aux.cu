// aux.cu -- initial state, macroscopic fields, population I/O and the wall Nusselt reduction.
#include <algorithm>

#include "kernels.h"
#include "step_d2q9.cuh"
#include "step_d3q27.cuh"

namespace lbm {

size_t storage_bytes(int prec)
{
    return prec == kF64 ? 8 : (prec == kF32 ? 4 : 2);
}

cudaError_t launch_step(int dim, int prec, const void* fin, const void* gin, void* fout, void* gout,
                        const Geometry& geo, const HostCoeffs& hc, unsigned* status, dim3 block,
                        bool flip, cudaStream_t st, const TmaMaps* tma)
{
    flip = flip && flip_pays(geo, dim == 2 ? 18 : 42, prec);
    if (dim == 2) return launch_step_d2q9(prec, fin, gin, fout, gout, geo, hc, status, block, flip, st);
    if (tma && prec == kF32) return launch_step_d3q27_tma_f32(*tma, fin, gin, fout, gout, geo, hc, status, st);
    if (tma && prec == kF16S) return launch_step_d3q27_tma_f16s(*tma, fin, gin, fout, gout, geo, hc, status, st);
    switch (prec) {
    case kF64: return launch_step_d3q27_f64(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    case kF32: return launch_step_d3q27_f32(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    case kF16S: return launch_step_d3q27_f16s(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    }
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------------------------
// Conversions between storage and double (F32 and F16S store deviations from the rest state;
// the full value shift + deviation is formed in double).
// ---------------------------------------------------------------------------------------------
// float -> double without the conversion instruction, which takes an FP64 pipe slot (16 cycles of an SM
// per warp, like an addition, even when predicated off), and that pipe bounds these passes.  A
// subnormal is first scaled by 2^24; infinities and NaN get the wider exponent.
__device__ __forceinline__ double widen(float v)
{
    const bool sub = (__float_as_uint(v) & 0x7f800000u) == 0u;
    const unsigned x = __float_as_uint(sub ? v * 16777216.0f : v), m = x & 0x7fffffffu;
    const unsigned bias = sub ? 0x36800000u : (m >= 0x7f800000u ? 0x70000000u : 0x38000000u);
    const unsigned hi = m == 0u ? 0u : (m >> 3) + bias;
    return __hiloint2double((int)((x & 0x80000000u) | hi), (int)(x << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

// A division out of line: inlined, its operations would take FP64 pipe slots in every warp even where no
// lane divides (160^3 FP32 fields 547 us against 132).
__device__ __noinline__ double divide(double a, double b) { return a / b; }

// By the bits: 2^-e <= |v| < 2^(e + 1); for e = 1023, every finite v.
__device__ __forceinline__ bool binary_exponent_within(double v, int e)
{
    const int b = (int)((unsigned)__double2hiint(v) >> 20 & 0x7ffu);
    return b >= 1023 - e && b <= 1023 + e;
}

template <class S> struct Conv;
template <> struct Conv<StoreF64> {
    __device__ static double get(double v, double) { return v; }
    __device__ static void put(double* p, size_t i, double v, double) { p[i] = v; }
};
template <> struct Conv<StoreF32> {
    __device__ static double get(float v, double s) { return s + widen(v); }
    __device__ static void put(float* p, size_t i, double v, double s) { p[i] = (float)(v - s); }
};
template <> struct Conv<StoreF16S> {
    // (the scale is a power of two: exact in FP32)
    __device__ static double get(__half v, double s) { return s + widen(__half2float(v) * StoreF16S::kInvScale); }
    __device__ static void put(__half* p, size_t i, double v, double s)
    {
        p[i] = __double2half((v - s) * (double)StoreF16S::kScale);
    }
};

template <int DIM> struct Lat;
template <> struct Lat<2> {
    static constexpr int QF = 9, QG = 9;
    __host__ __device__ static double wf(int a) { return w9(a); }
    __host__ __device__ static double wg(int a) { return w9(a); }
};
template <> struct Lat<3> {
    static constexpr int QF = 27, QG = 15;
    __host__ __device__ static double wf(int a) { return w27(a); }
    __host__ __device__ static double wg(int a) { return w15(a); }
};

// splitmix64 (Steele, Lea and Flood 2014): output i of the stream whose state starts at seed.
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t i)
{
    uint64_t z = seed + (i + 1) * 0x9e3779b97f4a7c15ULL;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

// Fluid at rest at density 1 and temperature T_init + perturb (2 U_i - 1); the populations are
// the rest attractors (the lattice weights times rho or T).
template <class S, int DIM>
__global__ void init_kernel(typename S::T* f, typename S::T* g, Geometry geo, double T_init,
                            double T_ref, uint64_t seed, double perturb)
{
    using L = Lat<DIM>;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < geo.n;
         i += (long long)gridDim.x * blockDim.x) {
        double T = T_init;
        if (perturb != 0.0) {
            const double u01 = (double)(splitmix64(seed, (uint64_t)i) >> 11) * (1.0 / 9007199254740992.0);
            T += perturb * (2.0 * u01 - 1.0);
        }
        for (int a = 0; a < L::QF; ++a) Conv<S>::put(f, (size_t)a * geo.n + i, L::wf(a), L::wf(a));
        for (int b = 0; b < L::QG; ++b)
            Conv<S>::put(g, (size_t)b * geo.n + i, L::wg(b) * T, L::wg(b) * T_ref);
    }
}

// Rest values of all planes, flow then energy (w_a and w_b T_ref), formed on the host.
struct PlaneShifts {
    double v[42];
};

// Population I/O: one plane per blockIdx.y, kIoRows elements per thread in flight.  One FP64 operation
// per element is left for FP32 and FP16 storage (the shift), so reading 160^3 FP32 takes 338 us against 642 with
// one node of every plane per thread and the conversions on the FP64 pipe (the HBM floor is 303).
constexpr int kIoRows = 4;

template <class S, int QF>
__global__ void __launch_bounds__(256)
    get_pops_kernel(const typename S::T* __restrict__ f, const typename S::T* __restrict__ g, long long n,
                    PlaneShifts shift, double* __restrict__ fo, double* __restrict__ go)
{
    const int a = blockIdx.y;
    const typename S::T* src = a < QF ? f + (size_t)a * n : g + (size_t)(a - QF) * n;
    double* dst = a < QF ? fo + (size_t)a * n : go + (size_t)(a - QF) * n;
    const double s = shift.v[a];
    const long long i0 = (long long)blockIdx.x * (256 * kIoRows) + threadIdx.x;
    typename S::T v[kIoRows];
#pragma unroll
    for (int r = 0; r < kIoRows; ++r)
        if (i0 + 256 * r < n) v[r] = src[i0 + 256 * r];
#pragma unroll
    for (int r = 0; r < kIoRows; ++r)
        if (i0 + 256 * r < n) dst[i0 + 256 * r] = Conv<S>::get(v[r], s);
}

template <class S, int QF>
__global__ void __launch_bounds__(256)
    set_pops_kernel(typename S::T* __restrict__ f, typename S::T* __restrict__ g, long long n, PlaneShifts shift,
                    const double* __restrict__ fi, const double* __restrict__ gi)
{
    const int a = blockIdx.y;
    typename S::T* dst = a < QF ? f + (size_t)a * n : g + (size_t)(a - QF) * n;
    const double* src = a < QF ? fi + (size_t)a * n : gi + (size_t)(a - QF) * n;
    const double s = shift.v[a];
    const long long i0 = (long long)blockIdx.x * (256 * kIoRows) + threadIdx.x;
    double v[kIoRows];
#pragma unroll
    for (int r = 0; r < kIoRows; ++r)
        if (i0 + 256 * r < n) v[r] = src[i0 + 256 * r];
#pragma unroll
    for (int r = 0; r < kIoRows; ++r)
        if (i0 + 256 * r < n) Conv<S>::put(dst, i0 + 256 * r, v[r], s);
}

// Streamed populations at one node as deviations from the rest state (the pull of the step
// kernels, without the collision).
template <class S, int DIM>
__device__ __forceinline__ void pulled(const typename S::T* f, const typename S::T* g,
                                       const Geometry& geo, typename S::R T_ref, int x, int y, int z,
                                       typename S::R* fo, typename S::R* go)
{
    using R = typename S::R;
    if constexpr (DIM == 2) {
        const NodeWalls<R> w = node_walls<R>(geo, x, y, 0, 2);
        pull_d2q9<S>(f, g, geo, w, x + geo.nx * y, T_ref, fo, go);
    } else {
        const NodeWalls<R> w = node_walls<R>(geo, x, y, z, 3);
        pull_d3q27_d3q15<S>(f, g, geo, w, x + geo.nx * y + geo.nxy * z, T_ref, fo, go);
    }
}

// Lattice velocity component d of link a.
template <int DIM>
__host__ __device__ constexpr int ev(int a, int d)
{
    if constexpr (DIM == 2) return e9(a, d);
    else return e27(a, d);
}

// Streamed deviations at one node, the pull chosen per warp as in the steps: interior rows without any
// wall bookkeeping.
template <class S, int DIM, class Idx>
__device__ __forceinline__ void pulled_by_warp(const typename S::T* f, const typename S::T* g, const Geometry& geo,
                                               typename S::R T_ref, int x, int y, int z, int i,
                                               typename S::R* fo, typename S::R* go)
{
    using R = typename S::R;
    const bool in = x > 0 && x < geo.nx - 1 && y > 0 && y < geo.ny - 1 && (DIM == 2 || (z > 0 && z < geo.nz - 1));
    if (__all_sync(__activemask(), in)) {
        if constexpr (DIM == 2) pull_d2q9_interior<S, Idx>(f, g, geo, i, T_ref, fo, go);
        else pull_d3q27_d3q15_interior<S, Idx>(f, g, geo, i, T_ref, fo, go);
    } else {
        const NodeWalls<R> w = node_walls<R>(geo, x, y, z, DIM);
        if constexpr (DIM == 2) pull_d2q9<S, Idx>(f, g, geo, w, i, T_ref, fo, go);
        else pull_d3q27_d3q15<S, Idx>(f, g, geo, w, i, T_ref, fo, go);
    }
}

// rho, u and T at every node (App. A Step 7, App. B Step 7, Sec. 6.1 force); a null output is not
// written, and kFlow = false (only T asked for) does not read the flow.  The sums run over the pulled
// deviations in the storage's register type (FP32 for FP32 and FP16 storage, where an FP64 sum made
// this pass bound by the FP64 pipe) and are promoted to FP64 for the outputs; there, too, FP64
// operations are what remains to save: widen() and one reciprocal for the three divisions (for FP32
// and FP16 storage within two ulps of FP64, on values that carry FP32 rounding).  Where that is no
// ordinary number (a diverged node's density 0, infinite or NaN) the velocity is the division's.  160^3: FP32 133 us against 644 (floor 125), T alone 69
// against 228; FP64 1067 against 1622.
template <class S, int DIM, class Idx, bool kFlow, bool kFlat>
__global__ void __launch_bounds__(256)
    fields_kernel(const typename S::T* f, const typename S::T* g, Geometry geo, double gbeta, double T_ref,
                  int gaxis, double* rho, double* ux, double* uy, double* uz, double* Tout)
{
    using R = typename S::R;
    using L = Lat<DIM>;
    int x, y, z, i;
    if constexpr (kFlat) {
        const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
        if (t >= (unsigned)geo.n) return;
        i = (int)t;
        z = DIM == 2 ? 0 : i / geo.nxy;
        const int r = i - z * geo.nxy;
        y = r / geo.nx;
        x = r - y * geo.nx;
    } else {
        x = blockIdx.x * blockDim.x + threadIdx.x;
        y = blockIdx.y * blockDim.y + threadIdx.y;
        z = blockIdx.z;
        if (x >= geo.nx || y >= geo.ny) return;
        i = x + geo.nx * y + geo.nxy * z;
    }
    R fo[L::QF], go[L::QG];
    pulled_by_warp<S, DIM, Idx>(f, g, geo, R(T_ref), x, y, z, i, fo, go);
    R dT = go[0];
    static_for<L::QG - 1>([&](auto B) { dT += go[decltype(B)::value + 1]; });
    const double dTd = widen(dT);
    if (Tout) Tout[i] = T_ref + dTd;
    if constexpr (kFlow) {
        R drho, j[3] = {R(0), R(0), R(0)};
        if constexpr (DIM == 3 && std::is_same<S, StoreF64>::value) {
            // FP64: over the raw x lines, half the additions
            R p[3][3][3];
            xraw_d3q27(fo, p);
            drho = R(0);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const R layer = (p[k][0][0] + p[k][2][0]) + p[k][1][0];
                drho += layer;
                if (k != 1) j[2] += k == 2 ? layer : -layer;
                j[1] += p[k][2][0] - p[k][0][0];
                j[0] += (p[k][0][1] + p[k][2][1]) + p[k][1][1];
            }
        } else {
            drho = fo[0];
            static_for<L::QF - 1>([&](auto A) {
                constexpr int a = decltype(A)::value + 1;
                drho += fo[a];
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    if (ev<DIM>(a, d) == 1) j[d] += fo[a];
                    if (ev<DIM>(a, d) == -1) j[d] -= fo[a];
                }
            });
        }
        const double r = 1.0 + widen(drho);
        const double hF = 0.5 * (gbeta * dTd);
        const double ir = recip(r);
        const bool ordinary = binary_exponent_within(r, 1000);   // and with it the reciprocal
        double* const out[3] = {ux, uy, uz};
        if (rho) rho[i] = r;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (!out[d]) continue;
            const double m = (d < DIM ? widen(j[d]) : 0.0) + (d == gaxis ? hF : 0.0);
            double q = m * ir;
            bool take = ordinary;
            if constexpr (std::is_same<S, StoreF64>::value) {
                // FP64 storage: one correction by the residual (Markstein 1990), which rounds as the
                // division does unless the quotient lies within 2^-50 of a tie
                take = take && binary_exponent_within(q, 1023);
                q = fma(fma(-q, r, m), ir, q);
            }
            out[d][i] = take ? q : divide(m, r);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Wall Nusselt number (Sec. 6.1): dT/dn = -8/3 T_w + 3 T_1 - 1/3 T_2 from the wall and the first
// two node layers; Nu = scale * dT/dn with scale = -s L / dT.  One thread per wall node, then
// FP64 warp-shuffle reductions of (sum, max with index, min with index), per-block partials and a
// final pass by the last block to finish (deterministic order, ties to the lowest index); a face of
// one block needs neither.
// ---------------------------------------------------------------------------------------------
// Extrema are kept as integer keys in the order of the values: an FP64 comparison takes an FP64 pipe slot,
// and the reductions are chains of them.  A NaN counts for neither (its keys lie beyond the infinities').
struct NuAcc {
    double sum;
    long long mx, mn;
    int imx, imn;
};

__device__ __forceinline__ long long nu_key(double v)
{
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double nu_value(long long k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}
// the neutral element: sum 0, max -inf, min +inf at no node
__device__ __forceinline__ NuAcc nu_none()
{
    return NuAcc{0.0, nu_key(-INFINITY), nu_key(INFINITY), 0x7fffffff, 0x7fffffff};
}
__device__ __forceinline__ NuAcc nu_node(double nu, int t)
{
    const bool nan = (__double_as_longlong(nu) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
    const long long k = nu_key(nu);
    return NuAcc{nu, nan ? nu_key(-INFINITY) : k, nan ? nu_key(INFINITY) : k, nan ? 0x7fffffff : t, nan ? 0x7fffffff : t};
}

__device__ __forceinline__ void nu_merge(NuAcc& a, const NuAcc& b)
{
    a.sum += b.sum;
    if (b.mx > a.mx || (b.mx == a.mx && b.imx < a.imx)) { a.mx = b.mx; a.imx = b.imx; }
    if (b.mn < a.mn || (b.mn == a.mn && b.imn < a.imn)) { a.mn = b.mn; a.imn = b.imn; }
}

__device__ __forceinline__ NuAcc nu_warp_reduce(NuAcc a)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        NuAcc b;
        b.sum = __shfl_down_sync(0xffffffffu, a.sum, o);
        b.mx = __shfl_down_sync(0xffffffffu, a.mx, o);
        b.mn = __shfl_down_sync(0xffffffffu, a.mn, o);
        b.imx = __shfl_down_sync(0xffffffffu, a.imx, o);
        b.imn = __shfl_down_sync(0xffffffffu, a.imn, o);
        nu_merge(a, b);
    }
    return a;
}

__device__ __forceinline__ NuAcc nu_block_reduce(NuAcc a)
{
    __shared__ NuAcc warp_part[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    a = nu_warp_reduce(a);
    if (lane == 0) warp_part[wid] = a;
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        // few warps: merged one after the other, no second tree
        if (nw <= 4) {
            for (int k = 1; k < nw; ++k) nu_merge(a, warp_part[k]);
        } else {
            a = nu_warp_reduce(lane < nw ? warp_part[lane] : nu_none());
        }
    }
    return a;
}

// The five result numbers {sum, max, argmax, min, argmin}.
__device__ __forceinline__ void nu_write(double* r, const NuAcc& a)
{
    r[0] = a.sum; r[1] = nu_value(a.mx); r[2] = (double)a.imx; r[3] = nu_value(a.mn); r[4] = (double)a.imn;
}

size_t nusselt_scratch_doubles(long n_face)
{
    const long nb = (n_face + 255) / 256;
    return (size_t)(5 * (nb < 1024 ? nb : 1024));
}

template <class S, int DIM>
__global__ void __launch_bounds__(256)
    nusselt_kernel(const typename S::T* f, const typename S::T* g, Geometry geo, double T_ref,
                   int face, int n_face, double scale, double* profile, double* partials,
                   unsigned* ticket, double* result)
{
    using R = typename S::R;
    using L = Lat<DIM>;
    const int ax = face >> 1, hi = face & 1;
    const int ext = ax == 0 ? geo.nx : (ax == 1 ? geo.ny : geo.nz);
    NuAcc acc = nu_none();
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n_face; t += gridDim.x * blockDim.x) {
        const int n0 = ax == 0 ? geo.ny : geo.nx;   // the faster of the face's two axes
        const int t1 = DIM == 2 ? 0 : t / n0, t0 = t - t1 * n0;
        R go[2][L::QG];
#pragma unroll
        for (int l = 0; l < 2; ++l) {   // both layers' loads in flight together
            const int c = hi ? ext - 1 - l : l;
            R fo[L::QF];
            pulled<S, DIM>(f, g, geo, R(T_ref), ax == 0 ? c : t0, ax == 0 ? t0 : (ax == 1 ? c : t1),
                           ax == 2 ? c : t1, fo, go[l]);
        }
        double Tl[2];
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            double s = 0.0;
#pragma unroll
            for (int b = 0; b < L::QG; ++b) s += widen(go[l][b]);
            Tl[l] = T_ref + s;
        }
        const int c = hi ? ext - 1 : 0;
        const double Tw = wall_temperature(geo, face, ax == 0 ? c : t0, ax == 0 ? t0 : (ax == 1 ? c : t1), ax == 2 ? c : t1);
        const double dTdn = -8.0 / 3.0 * Tw + 3.0 * Tl[0] - 1.0 / 3.0 * Tl[1];
        const double nu = scale * dTdn;
        profile[t] = nu;
        nu_merge(acc, nu_node(nu, t));
    }
    acc = nu_block_reduce(acc);
    if (gridDim.x == 1) {
        if (threadIdx.x == 0) nu_write(result, acc);
        return;
    }
    __shared__ bool last;
    if (threadIdx.x == 0) {
        nu_write(partials + 5 * blockIdx.x, acc);
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // Final pass: thread k takes partials k, k + blockDim, ... in order, then a block reduction.
    NuAcc tot = nu_none();
    for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) {
        const volatile double* p = partials + 5 * k;
        nu_merge(tot, NuAcc{p[0], nu_key(p[1]), nu_key(p[3]), (int)p[2], (int)p[4]});
    }
    tot = nu_block_reduce(tot);
    if (threadIdx.x == 0) {
        nu_write(result, tot);
        *ticket = 0u;
    }
}

// ---------------------------------------------------------------------------------------------
// Dispatch
// ---------------------------------------------------------------------------------------------
static int grid_for(long long n)
{
    long long b = (n + 255) / 256;
    return (int)(b < 65535 ? (b < 1 ? 1 : b) : 65535);
}

#define LBM_DISPATCH(dim, prec, ...)                                                   \
    do {                                                                                \
        if (dim == 2 && prec == kF64) { using S = StoreF64; constexpr int D = 2; __VA_ARGS__; } \
        else if (dim == 2 && prec == kF32) { using S = StoreF32; constexpr int D = 2; __VA_ARGS__; } \
        else if (dim == 2 && prec == kF16S) { using S = StoreF16S; constexpr int D = 2; __VA_ARGS__; } \
        else if (dim == 3 && prec == kF64) { using S = StoreF64; constexpr int D = 3; __VA_ARGS__; } \
        else if (dim == 3 && prec == kF32) { using S = StoreF32; constexpr int D = 3; __VA_ARGS__; } \
        else if (dim == 3 && prec == kF16S) { using S = StoreF16S; constexpr int D = 3; __VA_ARGS__; } \
        else return cudaErrorInvalidValue;                                              \
    } while (0)

cudaError_t launch_init(int dim, int prec, void* f, void* g, const Geometry& geo, double T_init,
                        double T_ref, uint64_t seed, double perturb, cudaStream_t st)
{
    LBM_DISPATCH(dim, prec, {
        using T = typename S::T;
        init_kernel<S, D><<<grid_for(geo.n), 256, 0, st>>>((T*)f, (T*)g, geo, T_init, T_ref, seed,
                                                           perturb);
    });
    return cudaGetLastError();
}

template <int DIM>
static PlaneShifts plane_shifts(double T_ref)
{
    using L = Lat<DIM>;
    PlaneShifts s{};
    for (int a = 0; a < L::QF; ++a) s.v[a] = L::wf(a);
    for (int b = 0; b < L::QG; ++b) s.v[L::QF + b] = L::wg(b) * T_ref;
    return s;
}

cudaError_t launch_get_pops(int dim, int prec, const void* f, const void* g, const Geometry& geo,
                            double T_ref, double* fo, double* go, cudaStream_t st)
{
    LBM_DISPATCH(dim, prec, {
        using T = typename S::T;
        const dim3 grid((unsigned)(((long long)geo.n + 256 * kIoRows - 1) / (256 * kIoRows)), Lat<D>::QF + Lat<D>::QG, 1);
        get_pops_kernel<S, Lat<D>::QF><<<grid, 256, 0, st>>>((const T*)f, (const T*)g, geo.n, plane_shifts<D>(T_ref),
                                                             fo, go);
    });
    return cudaGetLastError();
}

cudaError_t launch_set_pops(int dim, int prec, void* f, void* g, const Geometry& geo, double T_ref,
                            const double* fi, const double* gi, cudaStream_t st)
{
    LBM_DISPATCH(dim, prec, {
        using T = typename S::T;
        const dim3 grid((unsigned)(((long long)geo.n + 256 * kIoRows - 1) / (256 * kIoRows)), Lat<D>::QF + Lat<D>::QG, 1);
        set_pops_kernel<S, Lat<D>::QF><<<grid, 256, 0, st>>>((T*)f, (T*)g, geo.n, plane_shifts<D>(T_ref), fi, gi);
    });
    return cudaGetLastError();
}

template <class S, int D, class Idx>
static auto fields_instance(bool flow, bool flat)
{
    if (flat) return flow ? fields_kernel<S, D, Idx, true, true> : fields_kernel<S, D, Idx, false, true>;
    return flow ? fields_kernel<S, D, Idx, true, false> : fields_kernel<S, D, Idx, false, false>;
}

// Threads of the read-out along the linear index instead of along rows, where rows leave lanes idle: an idle
// lane costs as much as a busy one on the FP64 pipe and on the way to memory.  A warp that spans rows
// takes the general pull, which FP64, bound by its pipe, does not feel; 3D FP32 and FP16 do, the more
// of a row's warps would have been interior ones, and 2D a little.  All fields, a million nodes in 3D,
// 300,000 in 2D, rows -> flat: FP64 nx = 4 2315 -> 306 us, 33 543 -> 294, 100 348 -> 269, 150 276 -> 254, 250
// even; 3D FP32 4 298 -> 58, 33 84 -> 57, 40 77 -> 60, but 48 51 -> 56, 65 51 -> 54, 160 39 -> 53; 2D FP32 33
// 21 -> 12.6, 129 14.6 -> 12.5, 300 even (T alone 4.4 -> 5.2).
static bool fields_flat(const Geometry& g, int prec, int dim)
{
    const int lanes = (g.nx + 31) / 32 * 32, idle = lanes - g.nx;
    return (prec == kF64 ? 32 : (dim == 2 ? 8 : 3)) * idle > lanes;
}

cudaError_t launch_fields(int dim, int prec, const void* f, const void* g, const Geometry& geo,
                          const HostCoeffs& hc, double* rho, double* ux, double* uy, double* uz,
                          double* T, cudaStream_t st)
{
    const bool flat = fields_flat(geo, prec, dim);
    const dim3 b = flat ? dim3(256, 1, 1) : block_shape(geo, prec, dim);
    const dim3 grid = flat ? dim3((unsigned)(((long long)geo.n + 255) / 256), 1, 1) : grid_shape(geo, b);
    const bool flow = rho || ux || uy || uz;
    LBM_DISPATCH(dim, prec, {
        using TT = typename S::T;
        auto kern = index32(geo, Lat<D>::QF) ? fields_instance<S, D, unsigned>(flow, flat)
                                             : fields_instance<S, D, size_t>(flow, flat);
        kern<<<grid, b, 0, st>>>((const TT*)f, (const TT*)g, geo, hc.gbeta, hc.T_ref, hc.gaxis, rho, ux, uy, uz, T);
    });
    return cudaGetLastError();
}

bool host_writes()
{
    int dev = 0, v = 0, w = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrPageableMemoryAccess, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&w, cudaDevAttrPageableMemoryAccessUsesHostPageTables, dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return v != 0 && w != 0;
}

cudaError_t launch_nusselt(int dim, int prec, const void* f, const void* g, const Geometry& geo,
                           const HostCoeffs& hc, int face, double scale, double* profile,
                           double* scratch, unsigned* ticket, double* result, cudaStream_t st)
{
    const int ax = face >> 1;
    const long n_face = ax == 0 ? (long)geo.ny * geo.nz : (ax == 1 ? (long)geo.nx * geo.nz
                                                                    : (long)geo.nx * geo.ny);
    const int nb = (int)(nusselt_scratch_doubles(n_face) / 5);
    const int threads = (int)std::min<long>(256, (n_face + 31) / 32 * 32);
    LBM_DISPATCH(dim, prec, {
        using T = typename S::T;
        nusselt_kernel<S, D><<<nb, threads, 0, st>>>((const T*)f, (const T*)g, geo, hc.T_ref, face,
                                                 (int)n_face, scale, profile, scratch, ticket, result);
    });
    return cudaGetLastError();
}

}  // namespace lbm

// step2d.cu -- instantiations of the fused D2Q9 flow + D2Q9 energy step.
#include "kernels.h"
#include "step_d2q9.cuh"

namespace lbm {

constexpr int kPairNodes = 300000;  // nodes from which FP16 storage takes the pair kernel
constexpr int kSplitWarps = 448;   // warps of 32 nodes up to which FP64 boxes take the split kernel

template <class S, bool kUnit>
static cudaError_t run_as(const void* fin, const void* gin, void* fout, void* gout, const Geometry& geo,
                          const HostCoeffs& hc, unsigned* status, dim3 block, bool flip, cudaStream_t st)
{
    using T = typename S::T;
    using R = typename S::R;
    const int prec = std::is_same<S, StoreF64>::value ? kF64 : (std::is_same<S, StoreF32>::value ? kF32 : kF16S);
    const dim3 b = block_shape(geo, prec, 2, block);
    const dim3 grid((geo.nx + b.x - 1) / b.x, (geo.ny + b.y - 1) / b.y, 1);
    StepCoeffs2D<S, kUnit> c;
    if constexpr (kUnit) c = make_unit_coeffs<R, 2>(hc);
    else c = make_coeffs<R, 9, 9>(hc);
    auto kern = step_index32(geo, 9, hc) ? step_d2q9_kernel<S, unsigned, kUnit> : step_d2q9_kernel<S, size_t, kUnit>;
    return launch_step_kernel(kern, grid, b, st, (const T*)fin, (const T*)gin, (T*)fout, (T*)gout, geo, c, status,
                              flip);
}

template <class S>
static cudaError_t run(const void* fin, const void* gin, void* fout, void* gout, const Geometry& geo,
                       const HostCoeffs& hc, unsigned* status, dim3 block, bool flip, cudaStream_t st)
{
    if constexpr (std::is_same<S, StoreF64>::value) {
        // two warps per 32 nodes where they find a sub-partition each (112^2: 7.4 us against 7.6; 128^2: 8.7
        // against 8.3)
        const int bx = (geo.nx + 31) / 32;
        if (unit_rates_2d(hc) && block.x == 0 && (long long)bx * geo.ny <= kSplitWarps && step_index32(geo, 9, hc))
            return launch_step_kernel(step_d2q9_split_f64_kernel<unsigned>, dim3(bx, geo.ny, 1), dim3(64, 1, 1), st,
                                      (const double*)fin, (const double*)gin, (double*)fout, (double*)gout, geo,
                                      make_unit_coeffs<double, 2>(hc), status);
    }
    if constexpr (std::is_same<S, StoreF16S>::value) {
        // two nodes per thread where rows start on 4 bytes and fill its warps, in boxes that fill the SMs with them
        const bool aligned = (((uintptr_t)fin | (uintptr_t)gin | (uintptr_t)fout | (uintptr_t)gout) & 3) == 0;
        const bool filled = flip_pays(geo, 18, kF16S) ? pairs_fill_rows(geo.nx, 8, 5) : pairs_fill_rows(geo.nx, 15, 8);
        if (unit_rates_2d(hc) && block.x == 0 && geo.n >= kPairNodes && filled && aligned && step_index32(geo, 9, hc)) {
            // (blocks one warp wide where a row's warps are odd in number: nx = 192, 1.2 million nodes 17.5 -> 17.0 us)
            const bool odd = (geo.nx / 2 + 31) / 32 % 2 != 0;
            const dim3 b(odd ? 32 : 64, odd ? 4 : 2, 1);
            return launch_step_kernel(step_d2q9_pair_f16s_kernel<unsigned>, dim3((geo.nx / 2 + b.x - 1) / b.x, (geo.ny + b.y - 1) / b.y, 1),
                                      b, st, (const __half*)fin, (const __half*)gin, (__half*)fout, (__half*)gout, geo,
                                      make_unit_coeffs<float, 2>(hc), status, flip);
        }
    }
    if constexpr (has_unit_step<S>::value) {
        if (unit_rates_2d(hc)) return run_as<S, true>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    }
    return run_as<S, false>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
}

cudaError_t launch_step_d2q9(int prec, const void* fin, const void* gin, void* fout, void* gout,
                             const Geometry& geo, const HostCoeffs& hc, unsigned* status,
                             dim3 block, bool flip, cudaStream_t st)
{
    switch (prec) {
    case kF64: return run<StoreF64>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    case kF32: return run<StoreF32>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    case kF16S: return run<StoreF16S>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lbm

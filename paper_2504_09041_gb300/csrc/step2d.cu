// step2d.cu -- instantiations of the fused D2Q9 flow + D2Q9 energy step.
#include "kernels.h"
#include "step_d2q9.cuh"

namespace lbm {

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

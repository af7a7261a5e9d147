// step2d.cu -- instantiations of the fused D2Q9 flow + D2Q9 energy step.
#include "kernels.h"
#include "step_d2q9.cuh"

namespace lbm {

template <class S, bool kUnit>
static cudaError_t run_as(const void* fin, const void* gin, void* fout, void* gout, const Geometry& geo,
                          const HostCoeffs& hc, unsigned* status, dim3 b, bool flip, cudaStream_t st)
{
    using T = typename S::T;
    using R = typename S::R;
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
    const int prec = std::is_same<S, StoreF64>::value ? kF64 : (std::is_same<S, StoreF32>::value ? kF32 : kF16S);
    const StepShape shape = step_shape(geo, prec, 2, hc, block, starts_on_words(fin, gin, fout, gout));
    const dim3 b = shape.block;
    if constexpr (std::is_same<S, StoreF64>::value) {
        if (shape.kind == kStepSplit)
            return launch_step_kernel(step_d2q9_split_f64_kernel<unsigned>, dim3((geo.nx + 31) / 32, geo.ny, 1), b, st,
                                      (const double*)fin, (const double*)gin, (double*)fout, (double*)gout, geo,
                                      make_unit_coeffs<double, 2>(hc), status);
    }
    if constexpr (std::is_same<S, StoreF16S>::value) {
        if (shape.kind == kStepPair)
            return launch_step_kernel(step_d2q9_pair_f16s_kernel<unsigned>,
                                      dim3((geo.nx / 2 + b.x - 1) / b.x, (geo.ny + b.y - 1) / b.y, 1), b, st,
                                      (const __half*)fin, (const __half*)gin, (__half*)fout, (__half*)gout, geo,
                                      make_unit_coeffs<float, 2>(hc), status, flip);
    }
    if constexpr (has_unit_step<S>::value) {
        if (unit_rates_2d(hc)) return run_as<S, true>(fin, gin, fout, gout, geo, hc, status, b, flip, st);
    }
    return run_as<S, false>(fin, gin, fout, gout, geo, hc, status, b, flip, st);
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

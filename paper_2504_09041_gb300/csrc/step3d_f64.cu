// step3d_f64.cu -- the fused D3Q27 flow + D3Q15 energy step with StoreF64 storage (one
// translation unit per storage type so that the three heavy instantiations compile in parallel).
#include "kernels.h"
#include "step_d3q27.cuh"

namespace lbm {

// kU: the collision instance for the rates (rate_class).
template <int kU>
static cudaError_t launch_plain_f64(const void* fin, const void* gin, void* fout, void* gout,
                                    const Geometry& geo, const HostCoeffs& hc, unsigned* status,
                                    dim3 block, bool flip, cudaStream_t st)
{
    using S = StoreF64;
    using T = typename S::T;
    using R = typename S::R;
    const dim3 b = block_shape(geo, kF64, 3, block);
    const auto c = make_step_coeffs<R, kU>(hc);
    auto kern = step_index32(geo, 27, hc) ? step_d3q27_kernel<S, unsigned, 1, kU> : step_d3q27_kernel<S, size_t, 1, kU>;
    kern<<<grid_shape(geo, b), b, 0, st>>>((const T*)fin, (const T*)gin, (T*)fout, (T*)gout, geo, c, status, flip);
    return cudaGetLastError();
}

cudaError_t launch_step_d3q27_f64(const void* fin, const void* gin, void* fout, void* gout,
                                  const Geometry& geo, const HostCoeffs& hc, unsigned* status,
                                  dim3 block, bool flip, cudaStream_t st)
{
    switch (rate_class(hc)) {
    case 3: return launch_plain_f64<3>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    case 2: return launch_plain_f64<2>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    case 1: return launch_plain_f64<1>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    }
    return launch_plain_f64<0>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
}

}  // namespace lbm

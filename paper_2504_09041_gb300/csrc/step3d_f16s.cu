// step3d_f16s.cu -- the fused D3Q27 flow + D3Q15 energy step with StoreF16S storage (one
// translation unit per storage type so that the three heavy instantiations compile in parallel).
#include <algorithm>

#include "kernels.h"
#include "step_d3q27_tma.cuh"

namespace lbm {

// kU: the collision instance for the rates (rate_class).
template <int kU>
static cudaError_t launch_plain_f16s(const void* fin, const void* gin, void* fout, void* gout,
                                  const Geometry& geo, const HostCoeffs& hc, unsigned* status,
                                  dim3 block, bool flip, cudaStream_t st)
{
    using S = StoreF16S;
    using T = typename S::T;
    using R = typename S::R;
    const StepShape shape = step_shape(geo, kF16S, 3, hc, block, starts_on_words(fin, gin, fout, gout));
    const dim3 b = shape.block;
    if constexpr (kU == 3) {
        if (shape.kind == kStepPair) {
            step_d3q27_pair_f16s_kernel<unsigned><<<dim3((geo.nx / 2 + b.x - 1) / b.x, geo.ny, geo.nz), b, 0, st>>>(
                (const T*)fin, (const T*)gin, (T*)fout, (T*)gout, geo, make_unit_coeffs<R, 3>(hc), status, flip);
            return cudaGetLastError();
        }
    }
    const auto c = make_step_coeffs<R, kU>(hc);
    const bool idx32 = step_index32(geo, 27, hc);
    const int rows = idx32 ? rows3d_for(hc) : 1;
    auto kern = !idx32 ? step_d3q27_kernel<S, size_t, 1, kU>
                : rows == 4 ? step_d3q27_kernel<S, unsigned, 4, kU>
                : rows == 2 ? step_d3q27_kernel<S, unsigned, 2, kU>
                            : step_d3q27_kernel<S, unsigned, 1, kU>;
    dim3 g = grid_shape(geo, b);
    g.y = (g.y + rows - 1) / rows;
    kern<<<g, b, 0, st>>>((const T*)fin, (const T*)gin, (T*)fout, (T*)gout, geo, c, status, flip);
    return cudaGetLastError();
}

cudaError_t launch_step_d3q27_f16s(const void* fin, const void* gin, void* fout, void* gout,
                                  const Geometry& geo, const HostCoeffs& hc, unsigned* status,
                                  dim3 block, bool flip, cudaStream_t st)
{
    switch (rate_class(hc)) {
    case 3: return launch_plain_f16s<3>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    case 2: return launch_plain_f16s<2>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    case 1: return launch_plain_f16s<1>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
    }
    return launch_plain_f16s<0>(fin, gin, fout, gout, geo, hc, status, block, flip, st);
}

template <int TY, int kU>
static cudaError_t launch_tma_f16s(const TmaMaps& tm, const void* fin, const void* gin, void* fout,
                                  void* gout, const Geometry& geo, const HostCoeffs& hc,
                                  unsigned* status, cudaStream_t st)
{
    using S = StoreF16S;
    using T = typename S::T;
    using R = typename S::R;
    using L = TmaLayout<T, TY>;
    const auto c = make_step_coeffs<R, kU>(hc);
    const int tiles_x = (geo.nx + kTmaTX - 1) / kTmaTX, tiles_y = (geo.ny + TY - 1) / TY;
    const int n_tiles = tiles_x * tiles_y * geo.nz;
    const dim3 block(kTmaTX * TY + 32, 1, 1);   // TY rows of consumers and one producer warp
    auto kern = step_index32(geo, 27, hc) ? step_d3q27_tma_kernel<S, unsigned, TY, kU>
                                          : step_d3q27_tma_kernel<S, size_t, TY, kU>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kSmemBytes);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kTmaTX * TY + 32, L::kSmemBytes)) != cudaSuccess)
        return e;
    const int grid = std::max(1, std::min(n_tiles, sms * std::max(1, per_sm)));
    kern<<<grid, block, L::kSmemBytes, st>>>(tm.f, tm.g, (const T*)fin, (const T*)gin, (T*)fout, (T*)gout,
                                            geo, c, status, tiles_x, tiles_y, n_tiles);
    return cudaGetLastError();
}

template <int kU>
static cudaError_t launch_tma_rows_f16s(const TmaMaps& tm, const void* fin, const void* gin, void* fout,
                                       void* gout, const Geometry& geo, const HostCoeffs& hc,
                                       unsigned* status, cudaStream_t st)
{
    switch (tm.ty) {
    case 1: return launch_tma_f16s<1, kU>(tm, fin, gin, fout, gout, geo, hc, status, st);
    case 2: return launch_tma_f16s<2, kU>(tm, fin, gin, fout, gout, geo, hc, status, st);
    case 4: return launch_tma_f16s<4, kU>(tm, fin, gin, fout, gout, geo, hc, status, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_step_d3q27_tma_f16s(const TmaMaps& tm, const void* fin, const void* gin, void* fout,
                                      void* gout, const Geometry& geo, const HostCoeffs& hc,
                                      unsigned* status, cudaStream_t st)
{
    switch (rate_class(hc)) {
    case 3: return launch_tma_rows_f16s<3>(tm, fin, gin, fout, gout, geo, hc, status, st);
    case 2: return launch_tma_rows_f16s<2>(tm, fin, gin, fout, gout, geo, hc, status, st);
    case 1: return launch_tma_rows_f16s<1>(tm, fin, gin, fout, gout, geo, hc, status, st);
    }
    return launch_tma_rows_f16s<0>(tm, fin, gin, fout, gout, geo, hc, status, st);
}

}  // namespace lbm

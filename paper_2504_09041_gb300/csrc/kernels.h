// kernels.h -- host-side launchers of the CUDA kernels (internal to liblbm.so).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

#include <nvtx3/nvToolsExt.h>

#include "lattices.cuh"
#include "lbm_common.cuh"
#include "../../include/lbm.h"
#include <string>

namespace lbm {

// A named NVTX range on the calling thread's timeline for the duration of a library call
// (lbm_step, lbm_batch_step, lbm_adjoint_step): profilers that record NVTX show it above the
// kernels the call queued; without such a tool attached it costs two calls into a stub.
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

enum Prec { kF64 = 0, kF32 = 1, kF16S = 2 };

// Relaxation rates and coupling in double precision; converted to the kernel's register type.
struct HostCoeffs {
    double om_f[27];
    double om_g[15];
    double gbeta, T_ref;
    int gaxis;
    int gopt;   // energy attractors of orders 3-4: 0 = option A, 1 = option B
    int fp16_sr;   // F16S storage: stochastic (1) or nearest (0) rounding of stored deviations
    int index64;   // 1: the step uses 64-bit element offsets even where 32-bit ones suffice
    int rows3d;    // 3D FP32 / FP16S step: rows of its column each thread updates (1, 2 or 4; 0 automatic)
    int adj_sync;  // adjoint step blocks: 0 = 64x2; with phase barriers 1 = 64x4, 2 = 128x2 (default;
                   // 32x2 in large boxes), 3 = 32x4, 4 = 64x2
};

size_t storage_bytes(int prec);

// A validated box and its derived parameters (plan_box in api.cu).
struct BoxPlan {
    int lattice, prec, dim, nx, ny, nz, qf, qg;
    Geometry geo;
    HostCoeffs hc;
    double L, dT, U, nu, alpha;
};
int plan_box(int lattice, int nx, int ny, int nz, double Ra, double Pr, double Ma, const lbm_bc* bc,
             BoxPlan* P, std::string* err);
// Records the message of a failed call that has no handle (lbm_create, lbm_nusselt_static); lbm_last_error(NULL)
// returns it on the calling thread.  Returns code.
int fail_no_handle(int code, const char* fmt, ...);
// The process-wide device allocator hooks of lbm_set_allocator.
void current_allocator(lbm_alloc_fn* a, lbm_free_fn* f, void** ctx);

// Tensor maps of the input buffers of a TMA-staged 3D step (step_d3q27_tma.cuh) and its tile
// height (1, 2 or 4 rows of 64 nodes).
struct TmaMaps {
    CUtensorMap f, g;
    int ty;
};
// Encode the 4D map (x, y, z, plane) of one population buffer with boxes of (64 + 32 / elem_bytes)
// x ty x 1 x 1 elements.
// Fails (returns false, with a message) when the x stride is not a multiple of 16 bytes.
bool make_tma_map(CUtensorMap* out, void* base, int elem_bytes, int nx, int ny, int nz, int planes,
                  int ty, std::string* err);

// block: thread-block shape of the step launch (x-major); block.x == 0 selects the default.
// tma: tensor maps of fin / gin for the TMA-staged 3D step (FP32 and FP16S), or nullptr.
// flip: walk the box from its end where flip_pays.  Callers alternate it from step to step; the results
// are the same.
cudaError_t launch_step(int dim, int prec, const void* fin, const void* gin, void* fout, void* gout,
                        const Geometry& geo, const HostCoeffs& hc, unsigned* status, dim3 block,
                        bool flip, cudaStream_t st, const TmaMaps* tma = nullptr);
cudaError_t launch_step_d3q27_tma_f32(const TmaMaps& tm, const void* fin, const void* gin, void* fout,
                                      void* gout, const Geometry& geo, const HostCoeffs& hc,
                                      unsigned* status, cudaStream_t st);
cudaError_t launch_step_d3q27_tma_f16s(const TmaMaps& tm, const void* fin, const void* gin, void* fout,
                                       void* gout, const Geometry& geo, const HostCoeffs& hc,
                                       unsigned* status, cudaStream_t st);
cudaError_t launch_step_d2q9(int prec, const void* fin, const void* gin, void* fout, void* gout,
                             const Geometry& geo, const HostCoeffs& hc, unsigned* status,
                             dim3 block, bool flip, cudaStream_t st);
cudaError_t launch_step_d3q27_f64(const void* fin, const void* gin, void* fout, void* gout,
                                  const Geometry& geo, const HostCoeffs& hc, unsigned* status,
                                  dim3 block, bool flip, cudaStream_t st);
cudaError_t launch_step_d3q27_f32(const void* fin, const void* gin, void* fout, void* gout,
                                  const Geometry& geo, const HostCoeffs& hc, unsigned* status,
                                  dim3 block, bool flip, cudaStream_t st);
cudaError_t launch_step_d3q27_f16s(const void* fin, const void* gin, void* fout, void* gout,
                                   const Geometry& geo, const HostCoeffs& hc, unsigned* status,
                                   dim3 block, bool flip, cudaStream_t st);

cudaError_t launch_init(int dim, int prec, void* f, void* g, const Geometry& geo, double T_init,
                        double T_ref, uint64_t seed, double perturb, cudaStream_t st);
cudaError_t launch_fields(int dim, int prec, const void* f, const void* g, const Geometry& geo,
                          const HostCoeffs& hc, double* rho, double* ux, double* uy, double* uz,
                          double* T, cudaStream_t st);
cudaError_t launch_get_pops(int dim, int prec, const void* f, const void* g, const Geometry& geo,
                            double T_ref, double* fo, double* go, cudaStream_t st);
cudaError_t launch_set_pops(int dim, int prec, void* f, void* g, const Geometry& geo, double T_ref,
                            const double* fi, const double* gi, cudaStream_t st);

// Local wall Nusselt numbers of a fixed-T face and their mean / max / min.
// scratch must hold nusselt_scratch_doubles(n_face) doubles plus one unsigned ticket (ticket
// must be zero on entry and is left zero on exit).  result receives
// {sum, max, argmax, min, argmin} as doubles.
// profile is device memory of the library (a caller's buffer gets a copy, which knows other GPUs and ends
// of allocations); result likewise, or host memory where host_writes() holds.
size_t nusselt_scratch_doubles(long n_face);
// Kernels of the current device may write ordinary host memory (the CPU's page tables serve the GPU, as
// on Grace-Blackwell): a few result numbers then need no copy of their own.
bool host_writes();
cudaError_t launch_nusselt(int dim, int prec, const void* f, const void* g, const Geometry& geo,
                           const HostCoeffs& hc, int face, double scale, double* profile,
                           double* scratch, unsigned* ticket, double* result, cudaStream_t st);

// Adjoint of the D2Q9 step (adjoint_d2q9.cuh): seed mu_{n+1} = dJ/dp for J = mean Nu on `face`
// (mu must be zeroed first), and one fused adjoint step mu_{k+1} -> mu_k from the state s_{k-1},
// adding the design-face wall-temperature gradient (FP64) to grad.  `arith` is the arithmetic of
// the vector-Jacobian products and of mu: FP32 (4-byte mu), FP64 or double-float (8-byte mu).
enum AdjointArith { kAdjF32 = 0, kAdjF64 = 1, kAdjDF = 2 };
cudaError_t launch_adjoint_seed(const Geometry& geo, int face, double scale, void* mu, int arith,
                                cudaStream_t st);
cudaError_t launch_adjoint_step_d2q9(int prec, int arith, const void* f_prev, const void* g_prev,
                                     const void* mu_in, void* mu_out, const Geometry& geo,
                                     const HostCoeffs& hc, int design_face, double* grad,
                                     cudaStream_t st);

}  // namespace lbm

namespace lbm {

// Launch of a kernel that calls wait_previous_step: its blocks may start while the kernel before it on
// the stream is still running (a predecessor that is no kernel is waited for as usual).
template <class... P, class... A>
inline cudaError_t launch_step_kernel(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args)
{
    cudaLaunchAttribute overlap{};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cfg.attrs = &overlap;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
    if (e != cudaSuccess) cudaGetLastError();   // reported here, not again by the next launch
    return e;
}

template <class R, int QF, int QG>
inline Coeffs<R, QF, QG> make_coeffs(const HostCoeffs& h)
{
    Coeffs<R, QF, QG> c{};
    for (int a = 0; a < QF; ++a) {
        c.om_f[a] = R(h.om_f[a]);
        c.hf[a] = R(1.0 - 0.5 * h.om_f[a]);
    }
    for (int b = 0; b < QG; ++b) c.om_g[b] = R(h.om_g[b]);
    c.gbeta = R(h.gbeta);
    c.T_ref = R(h.T_ref);
    c.gaxis = h.gaxis;
    c.gopt = h.gopt;
    c.fp16_sr = h.fp16_sr;
    return c;
}

template <class R, int DIM>
inline UnitCoeffs<R> make_unit_coeffs(const HostCoeffs& h)
{
    UnitCoeffs<R> c{};
    for (int a = 4; a < 10; ++a) c.kf[a - 4] = a < (DIM == 2 ? 9 : 27) ? R(1.0 - h.om_f[a]) : R(0);
    for (int b = 1; b < 4; ++b) c.kg[b - 1] = R(1.0 - h.om_g[b]);
    c.gbeta = R(h.gbeta);
    c.T_ref = R(h.T_ref);
    c.rest_T = c.T_ref;
    if constexpr (DIM == 3 && std::is_same<R, double>::value) {
        const int first[3] = {0, 1, 7};
        for (int k = 0; k < 3; ++k) c.rest_g[k] = w15(first[k]) * h.T_ref;
        // (a sum of 53-bit numbers within a factor of 64 of each other: exact in 64 bits and more)
        c.rest_T = (double)((long double)c.rest_g[0] + 6.0L * c.rest_g[1] + 8.0L * c.rest_g[2]);
    }
    c.fp16_sr = h.fp16_sr;
    return c;
}

// The coefficients of the 3D step's collision instance kU.
template <class R, int kU>
inline auto make_step_coeffs(const HostCoeffs& h)
{
    if constexpr (kU == 3) return make_unit_coeffs<R, 3>(h);
    else return make_coeffs<R, 27, 15>(h);
}

// Default thread blocks, x-major so that a warp reads and writes 32 consecutive nodes; a
// caller-chosen shape (block.x > 0) replaces it.
// 2D, FP64: one warp, so that few warps spread over all SMs: an SM takes one FP64 warp instruction per 16
//   cycles and a sub-partition one per 64, so 128^2 nodes (512 warps) take 8.4 us a step against 14.9 in
//   blocks of 256 threads on 64 SMs; 1024 x 512 takes 176.2 us against 181.8 (a finer tail).
//   Above 65535 rows two warps, the launch grid's limit.
// 2D, FP32 and FP16 storage: 64 x 2 (1024 x 512 FP32 9.91 us against 10.12 for 256 threads, 512^2 5.71
//   against 5.79, 64^2 1.71 against 1.98; one warp per block 10.5, bound by block turnover); 96 x 2 for
//   rows of three warps, of which 64 x 2 leaves a quarter idle (96 x 900 FP32 2.82 us against 3.21, 78 x 1406 3.66
//   against 4.53, 95 x 13000 29.9 against 31.2).
// 3D: 64 x 1, which at 72-96 registers per thread lets 10-14 blocks share an SM against four of 256
//   threads (256^3 FP32 837 us against 851); 32 x 1 where a row ends in a half-empty block
//   (131 x 93 x 77: FP32 65.3 us against 68.4, FP16S 45.8 against 53.5, FP64 1292 against 1306);
//   128 x 1 from two million nodes on, where rows fill such blocks (256^3: FP32 834 us against 837, FP16S one
//   node per thread 801 against 806; but 64^3 FP32 18.7 against 17.8, FP16S 16.3 against 14.6).  Above 65535 rows
//   two rows of them, as in 2D.
inline dim3 block_shape(const Geometry& g, int prec, int dim, dim3 chosen = dim3(0, 0, 0))
{
    if (chosen.x > 0) return dim3(chosen.x, chosen.y, 1);
    const int warps = (g.nx + 31) / 32;   // per row
    const int rows = g.ny > 65535 ? 2 : 1;
    if (dim == 3) return dim3(warps & 1 ? 32 : (warps & 3 || g.n < (1 << 21) ? 64 : 128), rows, 1);
    if (prec == kF64) return dim3(32, rows, 1);
    return warps == 1 ? dim3(32, 4, 1) : dim3(warps == 3 ? 96 : 64, 2, 1);
}

// 32-bit element offsets suffice when every population plane index q * n fits in 32 bits.
inline bool index32(const Geometry& g, int q)
{
    return (unsigned long long)q * (unsigned long long)g.n <= 0xffffffffULL;
}

// The step's offset width: 32-bit where q n < 2^32, unless the handle forces the 64-bit
// instantiation (which boxes above that size run; forcing it lets small boxes test it).
inline bool step_index32(const Geometry& g, int q, const HostCoeffs& hc)
{
    return index32(g, q) && !hc.index64;
}

// The energy rates are those lbm_create sets (option A; every rate 1 except the first-order ones,
// which carry alpha), so the 3D step may take the unit-rate energy collision.
inline bool unit_energy_rates(const HostCoeffs& h)
{
    if (h.gopt != 0) return false;
    for (int b = 4; b < 15; ++b)
        if (h.om_g[b] != 1.0) return false;
    return true;
}

// The 3D flow rates are those lbm_create sets: every rate 1 except the shear rates (slots 4-6,
// 8, 9), the bulk rate (slot 7) included.
inline bool unit_flow_rates(const HostCoeffs& h)
{
    for (int a = 0; a < 27; ++a)
        if (!(a >= 4 && a <= 6) && a != 8 && a != 9 && h.om_f[a] != 1.0) return false;
    return true;
}

// The 2D box takes the reduced collision (collide_store_d2q9_unit): option A, every rate 1 except the
// shear (flow slots 4, 5) and diffusivity (energy slots 1, 2) ones, gravity along y.
inline bool unit_rates_2d(const HostCoeffs& h)
{
    if (h.gopt != 0 || h.gaxis != 1) return false;
    for (int a = 0; a < 9; ++a)
        if ((a != 4 && a != 5 && h.om_f[a] != 1.0) || (a != 1 && a != 2 && h.om_g[a] != 1.0)) return false;
    return true;
}

// Which collision instance the 3D step takes: 0 general, 1 unit-rate energy collision, 2 that and
// the unit-rate flow relaxation, 3 that with gravity along z (collide_store_d3q27_unit; FP32 storage
// takes instance 2 there, see has_unit_step).
inline int rate_class(const HostCoeffs& h)
{
    if (!unit_energy_rates(h)) return 0;
    if (!unit_flow_rates(h)) return 1;
    return h.gaxis == 2 ? 3 : 2;
}

// Rows per thread of the 3D FP32 / FP16S step: the handle's setting, or when that is 0 one, the
// fastest with every collision (128^3 FP32 107 us against 113 for two rows, FP16S 82 against 85; 256^3 FP32 835
// against 850; only the general collision at 256^3 is within 0.2 % either way).
inline int rows3d_for(const HostCoeffs& h) { return h.rows3d > 0 ? h.rows3d : 1; }

// Both buffers of a box exceed the 129 MB L2.  A step that walks the box in the other direction than the one
// before it then starts with the rows written last, which are still there: 131 x 93 x 77 FP32 69.4 ->
// 62.8 us with option B, 128^3 113.5 -> 108.6, 256^3 831 -> 825 (default rates), 2048 x 1024 46.1 -> 44.1.
// Boxes that fit in L2 as a whole lose a little (64^3 14.5 -> 15.1 us, 1024 x 512 10.0 -> 10.2).
inline bool flip_pays(const Geometry& g, int q, int prec)
{
    return 2.0 * q * (double)g.n * (double)storage_bytes(prec) > 129e6;
}

// FP16 storage, two nodes per thread: rows must fill the pairs' warps about as well as they fill single
// nodes'.  A pair's warp does the work of num / den one-node warps:
// - 2D, both buffers in L2, 15 / 8: 1.2 million nodes, pairs against one node, nx = 64 17.5 us against 18.2, 128
//   16.3 against 17.7; but 32 33.0 against 18.2, 96 21.1 against 18.5, 160 20.5 against 18.1, 258 20.3 against 19.4.
// - 2D beyond, 8 / 5: 8 million, 64 114 against 124, 130 151 against 155, 322 119 against 139; but 96 133 against 129.
// - 3D, 7 / 4: 6.4 million, 98 336 against 343, 258 315 against 320; but 32 507 against 289, 96 339 against 287, 160 323
//   against 288, 194 339 against 328.
inline bool pairs_fill_rows(int nx, int num, int den)
{
    return nx % 2 == 0 && num * ((nx / 2 + 31) / 32) < den * ((nx + 31) / 32);
}

inline dim3 grid_shape(const Geometry& g, dim3 b)
{
    return dim3((g.nx + b.x - 1) / b.x, (g.ny + b.y - 1) / b.y, g.nz);
}

// Which step kernel a box takes, and its thread blocks; on_words: its buffers start on 4 bytes.
enum StepKind {
    kStepNode,    // one thread per node
    kStepSplit,   // 2D FP64: the two lattices of a node on two warps (step_d2q9_split_f64_kernel)
    kStepPair     // FP16 storage: two nodes per thread (step_d2q9_pair_f16s_kernel, step_d3q27_pair_f16s_kernel)
};
struct StepShape {
    StepKind kind;
    dim3 block;
};

constexpr int kPairNodes2D = 300000, kPairNodes3D = 6000000;   // nodes from which boxes fill the SMs with pairs
constexpr int kSplitWarps = 448;   // warps of 32 nodes up to which two warps per 32 nodes find a sub-partition each
                                   // (112^2: 7.4 us against 7.6; 128^2: 8.7 against 8.3)

inline StepShape step_shape(const Geometry& g, int prec, int dim, const HostCoeffs& hc, dim3 chosen, bool on_words)
{
    const bool reduced = dim == 2 ? unit_rates_2d(hc) : rate_class(hc) == 3;
    if (reduced && chosen.x == 0 && step_index32(g, dim == 2 ? 9 : 27, hc)) {
        if (dim == 2 && prec == kF64 && (long long)((g.nx + 31) / 32) * g.ny <= kSplitWarps)
            return {kStepSplit, dim3(64, 1, 1)};
        // pairs, one warp wide where a row's warps are odd in number (2D nx = 192, 1.2 million nodes 17.5 -> 17.0 us)
        const int odd = (g.nx / 2 + 31) / 32 % 2;
        if (dim == 2 && prec == kF16S && on_words && g.n >= kPairNodes2D &&
            (flip_pays(g, 18, prec) ? pairs_fill_rows(g.nx, 8, 5) : pairs_fill_rows(g.nx, 15, 8)))
            return {kStepPair, odd ? dim3(32, 4, 1) : dim3(64, 2, 1)};
        if (dim == 3 && prec == kF16S && on_words && g.n >= kPairNodes3D && hc.rows3d == 0 && g.ny <= 65535 &&
            pairs_fill_rows(g.nx, 7, 4))
            return {kStepPair, dim3(odd ? 32 : 64, 1, 1)};
    }
    return {kStepNode, block_shape(g, prec, dim, chosen)};
}

inline bool starts_on_words(const void* a, const void* b, const void* c, const void* d)
{
    return (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d) & 3) == 0;
}

}  // namespace lbm

"""Host code of the library against a fake CUDA runtime: what it does where a GPU would have to misbehave
to show it.  The programs hold no device code and run on the CPU."""
import os
import subprocess

import pytest

from paper_2504_09041_gb300 import build as B

# The fake runtime: an allocator on the host, and the registration calls that nvcc emits.
RUNTIME = r"""
#include <cstdio>
#include <cstdlib>
#include <cstdint>
#include <cuda_runtime_api.h>
#include "lbm.h"
extern "C" {
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction() {}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
}
"""


def run(tmp_path, name, source, objects=()):
    """Compile source against the library's translation units `objects`; the program's output."""
    nvcc = B._nvcc()
    include = [f"-I{p}" for p in (B.CSRC, os.path.join(B.HERE, "..", "include"),
                                  os.path.join(os.path.dirname(nvcc), "..", "include"))]
    main = tmp_path / (name + ".cpp")
    main.write_text(RUNTIME + source)
    exe = str(tmp_path / name)
    objs = []
    for src in objects:
        objs.append(str(tmp_path / (os.path.basename(src) + ".o")))
        subprocess.run([nvcc, *B.ARCH, "-O0", "-std=c++17", "--expt-relaxed-constexpr", *include, "-c",
                        os.path.join(B.CSRC, src), "-o", objs[-1]], check=True, timeout=300)
    # (calls of the runtime that the program does not reach stay unresolved)
    subprocess.run(["g++", "-std=c++17", *include, str(main), *objs, "-o", exe, "-ldl",
                    "-Wl,--unresolved-symbols=ignore-all"], check=True, timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    return r.stdout.split()


PROFILE = r"""
static int where;                 // device the caller's memory is said to be on
static double* kernel_dst;        // what the reduction kernel was given for the profile
static void* copy_dst;
static size_t copy_bytes;
namespace lbm {
struct Geometry;
struct HostCoeffs;
size_t storage_bytes(int) { return 8; }
size_t nusselt_scratch_doubles(long) { return 5; }
bool host_writes() { return false; }
cudaError_t launch_init(int, int, void*, void*, const Geometry&, double, double, uint64_t, double, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_nusselt(int, int, const void*, const void*, const Geometry&, const HostCoeffs&, int, double,
                           double* profile, double*, unsigned*, double*, cudaStream_t)
{
    kernel_dst = profile;
    return cudaSuccess;
}
}
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*)
{
    a->type = cudaMemoryTypeDevice;
    a->device = where;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void*, size_t n, cudaMemcpyKind, cudaStream_t)
{
    copy_dst = d;
    copy_bytes = n;
    return cudaSuccess;
}
}
int main()
{
    lbm_bc bc{{LBM_WALL_FIXED_T, LBM_WALL_FIXED_T, LBM_WALL_ADIABATIC, LBM_WALL_ADIABATIC, 0, 0}, {1, 0}, .5, .5, 1, 0, 0};
    lbm_handle h = nullptr;
    if (lbm_create(LBM_D2Q9_D2Q9 | LBM_FP64, 8, 6, 1, 1e4, 0.71, 0.1, &bc, &h) != LBM_OK) return 1;
    static double out[6];
    for (where = 0; where < 2; ++where) {
        copy_dst = nullptr;
        if (lbm_nusselt_profile(h, 0, out, 6, 1) != LBM_OK) return 2;
        printf("%d %d ", kernel_dst == out, copy_dst == out && copy_bytes == sizeof out);
    }
    return 0;
}
"""


def test_wall_profile_reaches_the_caller_by_a_copy(tmp_path):
    """The caller's pointer may name memory of another GPU, or less memory than the face needs: a copy
    serves the one and reports the other, a kernel's store does neither.  So the kernel writes memory of
    the handle and the copy goes to the caller, wherever the pointer is said to be."""
    assert run(tmp_path, "profile", PROFILE, ["api.cu"]) == ["0", "1", "0", "1"]


LAUNCH = r"""
static cudaError_t last = cudaSuccess;
extern "C" {
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**)
{
    return last = cudaErrorInvalidConfiguration;
}
cudaError_t cudaGetLastError()
{
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
int launch_nothing();
}
int main()
{
    const int e = launch_nothing();
    printf("%d %d", e == cudaErrorInvalidConfiguration, cudaGetLastError() == cudaSuccess);
    return 0;
}
"""


def test_failed_launch_leaves_no_error_behind(tmp_path):
    """The launch of a dependent step reports its own error once: the next good call, which ends in
    cudaGetLastError, must not report it again as its own."""
    kernel = tmp_path / "nothing.cu"
    kernel.write_text("""
#include "kernels.h"
__global__ void nothing(int) {}
extern "C" int launch_nothing() { return lbm::launch_step_kernel(nothing, dim3(1), dim3(1), nullptr, 3); }
""")
    assert run(tmp_path, "launch", LAUNCH, [str(kernel)]) == ["1", "1"]

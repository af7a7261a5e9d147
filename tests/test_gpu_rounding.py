"""Rounding of single operations and updates, where whole runs would hide it."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_09041_gb300 import build as B  # noqa: E402
from paper_2504_09041_gb300 import lbm as L  # noqa: E402


E15 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 1), (-1, 1, 1),
       (1, -1, 1), (-1, -1, 1), (1, 1, -1), (-1, 1, -1), (1, -1, -1), (-1, -1, -1)]


def energy_sum_drift(axis, T_lo, T_hi, T_ref):
    """RMS over the nodes of a periodic box of what one FP64 step adds to the sum of a node's energy
    populations, which the collision conserves.  The sums are formed in extended precision."""
    n = 32
    walls = L.Walls((L.LBM_PERIODIC,) * 6, (0,) * 6, T_ref, T_ref, axis)
    lat = L.Lattice("d3q27", n, n, n, Ra=1e5, walls=walls, precision="fp64")
    lat.set_param("gbeta", 0.0)
    rng = np.random.default_rng(11)
    f, g = lat.get_populations()
    e = np.array(E15)
    w = np.array([2 / 9] + [1 / 9] * 6 + [1 / 72] * 8)
    T = rng.uniform(T_lo, T_hi, g.shape[1:])
    u = rng.uniform(-0.06, 0.06, (3, *T.shape))
    g = w[:, None, None, None] * T * (1 + 3 * np.einsum("bd,dzyx->bzyx", e, u))
    lat.set_populations(f * (1 + 0.05 * rng.uniform(-1, 1, f.shape)), g)
    lat.step(1)
    lat.sync()
    _, after = lat.get_populations()
    lat.close()
    pulled = np.stack([np.roll(g[b], (e[b][2], e[b][1], e[b][0]), axis=(0, 1, 2)) for b in range(15)])
    d = after.astype(np.longdouble).sum(axis=0) - pulled.astype(np.longdouble).sum(axis=0)
    return float(np.sqrt((d * d).mean()))


@pytest.mark.parametrize("T_lo,T_hi,T_ref", [(0.0, 1.0, 0.5), (0.45, 0.55, 0.5), (0.9, 1.0, 0.5), (0.0, 1.0, 0.3),
                                             (20.0, 30.0, 25.0)])
def test_fp64_3d_energy_rounds_no_more_than_the_collision_it_replaces(T_lo, T_hi, T_ref):
    """Gravity along z takes the reduced step, along y the collision on deviations it replaces; without
    a force both compute the same function of the same state."""
    assert energy_sum_drift(2, T_lo, T_hi, T_ref) <= energy_sum_drift(1, T_lo, T_hi, T_ref)


RECIP = r"""
#include "lbm_common.cuh"
template <class R>
__global__ void recip_kernel(const R* x, R* y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = lbm::recip(x[i]);
}
extern "C" int recip64(const double* x, double* y, int n)
{
    recip_kernel<<<(n + 255) / 256, 256>>>(x, y, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int recip32(const float* x, float* y, int n)
{
    recip_kernel<<<(n + 255) / 256, 256>>>(x, y, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def recip_lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("recip")
    (d / "recip.cu").write_text(RECIP)
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-Xcompiler", "-fvisibility=default", "-I", B.CSRC, "-shared",
                    str(d / "recip.cu"), "-o", str(d / "recip.so")], check=True, timeout=300)
    return ctypes.CDLL(str(d / "recip.so"))


@pytest.mark.parametrize("dtype,call", [(np.float64, "recip64"), (np.float32, "recip32")])
@pytest.mark.parametrize("lo,hi", [(0.5, 2.0), (512.0, 2048.0), (1e-6, 1e6)])
def test_reciprocal_is_within_an_ulp(recip_lib, dtype, call, lo, hi):
    """Densities lie about 1, or about 1024 in the units of FP16 storage.  After the step the error is
    half an ulp of rounding and the residual's next order: with 20 bits of approximation 2^-60 for double,
    2^-40 for float; so the nearest number or a neighbour of it."""
    rng = np.random.default_rng(3)
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), 1 << 20)).astype(dtype)
    x[:2] = lo, hi
    t = torch.from_numpy(x).cuda()
    y = torch.empty_like(t)
    assert getattr(recip_lib, call)(ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(y.data_ptr()), x.size) == 0
    want = (1 / x.astype(np.longdouble)).astype(dtype)
    assert (np.abs(y.cpu().numpy() - want) <= np.spacing(want)).all()


def velocity_box(precision, f0, f1):
    """A periodic 2D box whose flow populations are at rest but for links 0 and 1; rho and u_x without a
    force, and the momentum of each node (link 1 comes from the node to the left)."""
    walls = L.Walls((L.LBM_PERIODIC,) * 6, (0,) * 6, 0.5, 0.5, 1)
    lat = L.Lattice("d2q9", f0.shape[1], f0.shape[0], Ra=1e4, walls=walls, precision=precision)
    lat.set_param("gbeta", 0.0)
    f, g = lat.get_populations()
    rest = f[1, 0, 0, 0]
    f[0, 0], f[1, 0] = f0, f1
    lat.set_populations(f, g)
    f, _ = lat.get_populations()            # as stored
    out = {k: v.cpu().numpy()[0] for k, v in lat.fields().items()}
    lat.close()
    j = f[1, 0] - rest
    if precision != "fp64":                 # (the stored deviation has at most 24 bits; reading it added the rest)
        j = j.astype(np.float32).astype(np.float64)
    return out["rho"], out["ux"], np.roll(j, 1, axis=1)


def test_fp64_velocity_is_the_division():
    """The corrected quotient rounds as the division unless it lies within 2^-50 of a tie between two
    numbers, which 10^6 nodes do not meet."""
    rng = np.random.default_rng(5)
    rho, ux, j = velocity_box("fp64", rng.uniform(0.2, 1.5, (1024, 1024)), rng.uniform(0.0, 0.3, (1024, 1024)))
    assert rho.min() > 0.6 and rho.max() < 2.4
    np.testing.assert_array_equal(ux, j / rho)


def test_fp32_velocity_is_within_two_ulps_of_the_division():
    """A reciprocal within 2^-53 of itself and one rounding: 2^-52 of the quotient, and the division's own
    half ulp."""
    rng = np.random.default_rng(6)
    rho, ux, j = velocity_box("fp32", rng.uniform(0.2, 1.5, (512, 512)), rng.uniform(0.0, 0.3, (512, 512)))
    assert (np.abs(ux - j / rho) <= 2 * np.spacing(np.abs(j / rho))).all() and np.abs(ux).max() > 0.01


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16s"])
def test_velocity_of_diverged_nodes(precision):
    """At density infinity, 0 or NaN the velocity is what the division gives: 0, an infinity, NaN."""
    n = 64
    f0 = np.full((1, n), 4 / 9)
    f0[0, 5], f0[0, 9], f0[0, 11] = np.inf, -np.inf, np.nan
    k = np.arange(n - 16)
    f0[0, 16:] = 4 / 9 - 1 - 0.125 + (k - 20) * 2.0 ** -56     # densities about 0, one of them exactly
    if precision != "fp64":
        f0[0, 16:] = 4 / 9 - 1 - 0.125
    rho, ux, j = velocity_box(precision, f0, np.full((1, n), 1 / 9 + 0.125))
    with np.errstate(divide="ignore", invalid="ignore"):
        want = j / rho
    assert ux[0, 5] == 0 and ux[0, 9] == 0 and np.isnan(ux[0, 11])
    zero = rho[0] == 0
    assert zero.any() and np.isposinf(ux[0, zero]).all()
    np.testing.assert_allclose(ux, want, rtol=2.0 ** -51)

"""The adjoint step's block shapes agree, on both sides of the size where the default changes over, and
the reduced products of the default rates agree with the general ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_09041_gb300 import lbm as L  # noqa: E402


def gradient(nx, ny, precision="fp32", om0=None, steps=12, kind="cavity", **params):
    walls = L.Walls.cavity(2) if kind == "cavity" else L.Walls.rayleigh_benard(seed=3, perturb=0.05)
    faces = (1, 0) if kind == "cavity" else (3, 2)
    lat = L.Lattice("d2q9", nx, ny, Ra=1e5, walls=walls, precision=precision)
    if om0 is not None:
        inf = lat.info()
        om_f = np.array(inf.om_f[:9])
        om_f[0] = om0
        lat.set_omegas(om_f, np.array(inf.om_g[:9]))
    lat.set_param("gbeta", 3e-3)
    for k, v in params.items():
        lat.set_param(k, v)
    J, grad = lat.adjoint(steps, *faces)
    lat.close()
    return J, grad


# The shapes run the same products in the same order; the default's 32 x 2 blocks start at 305 blocks of
# 128 x 2 (the sizes straddle it and leave ragged ends).
@pytest.mark.parametrize("nx,ny", [(128, 608), (129, 306), (130, 609), (37, 611)])
def test_block_shapes_agree(nx, ny):
    J, grad = gradient(nx, ny)
    for sync in (4, 0):
        J2, g2 = gradient(nx, ny, adjoint_sync=sync)
        assert J2 == J
        # double-float values: a few 2^-48 per operation, some 10^3 operations deep
        assert np.abs(g2 - grad).max() <= 1e-10 * np.abs(grad).max()


# One rate moved by 1e-12 selects the general products; the zero terms they carry are then 1e-12 of their
# neighbours', and FP32 states do not move at all (1 - 1e-12 rounds to 1 in FP32).
@pytest.mark.parametrize("arith,tol", [(2, 1e-9), (1, 1e-9), (0, 1e-4)])
@pytest.mark.parametrize("kind,nx,ny", [("cavity", 40, 33), ("rb", 31, 20)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_reduced_products_equal_general_ones(precision, kind, nx, ny, arith, tol):
    J, grad = gradient(nx, ny, precision, kind=kind, steps=40, adjoint_arith=arith)
    J2, g2 = gradient(nx, ny, precision, om0=1.0 - 1e-12, kind=kind, steps=40, adjoint_arith=arith)
    assert J2 == pytest.approx(J, rel=1e-10)
    assert np.abs(g2 - grad).max() <= tol * np.abs(grad).max()

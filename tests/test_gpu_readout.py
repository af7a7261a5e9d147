"""Population and field read-out: every value of the storage type comes back exactly, and each field is
the same whether it is asked for alone or with the others."""
import numpy as np
import pytest

from tests import synth
from tests.test_gpu_parity import make_pair, randomize

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_09041_gb300 import lbm as L  # noqa: E402


@pytest.mark.parametrize("precision,store", [("fp32", np.float32), ("fp16s", np.float16), ("fp64", np.float64)])
@pytest.mark.parametrize("shape", [(1, 1), (31, 33), (32, 32), (25, 41)])
def test_populations_round_trip_special_values(precision, store, shape):
    """With T_ref = 0 the energy planes are stored as they are (FP16 storage: times 2^10), so what comes
    back is the stored number widened: exact, for zeros, subnormals, infinities and NaN too.  The sizes
    straddle the 1024 elements of a block."""
    ny, nx = shape
    walls = L.Walls((L.LBM_PERIODIC,) * 6, (0,) * 6, 0.0, 0.0, 1)
    lat = L.Lattice("d2q9", nx, ny, walls=walls, precision=precision)
    scale = 1024.0 if precision == "fp16s" else 1.0
    special = np.array([0.0, -0.0, 1e-40, -3e-42, 1.4e-45, 1.1754944e-38, 6e-8, -5.96e-8, 0.1, -1 / 3,
                        3.4e38, np.inf, -np.inf, np.nan])
    g = np.resize(special, (9, 1, ny, nx)).astype(np.float64)
    f, _ = lat.get_populations()
    lat.set_populations(f, g)
    fb, gb = lat.get_populations()
    lat.close()
    with np.errstate(over="ignore"):
        want = (g * scale).astype(store).astype(np.float64) / scale
    np.testing.assert_array_equal(gb, want)
    np.testing.assert_array_equal(np.signbit(gb[~np.isnan(gb) & (gb != 0)]), np.signbit(want[~np.isnan(gb) & (gb != 0)]))
    np.testing.assert_array_equal(fb, f)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16s"])
@pytest.mark.parametrize("lattice,shape", [("d2q9", (1, 9, 70)), ("d3q27", (5, 6, 33)), ("d3q27", (1, 2, 64))])
def test_fields_alone_equal_fields_together(lattice, shape, precision):
    nz, ny, nx = shape
    lat = L.Lattice(lattice, nx, ny, nz, Ra=1e4, precision=precision)
    f, g = lat.get_populations()
    lat.set_populations(synth.perturbed(f, 1, 0.05), synth.perturbed(g, 2, 0.05))
    lat.step(2)
    names = ("rho", "ux", "uy", "uz", "T")
    together = lat.fields()
    for k, name in enumerate(names):
        out = torch.full(lat.shape, float("nan"), dtype=torch.float64, device="cuda")
        L.lbm_fields(lat.h, *[out.data_ptr() if i == k else None for i in range(5)], 1)
        torch.cuda.synchronize()
        assert torch.equal(out, together[name]), name
    lat.close()


@pytest.mark.parametrize("lattice,shape,face", [("d2q9", (1, 1, 2), 0), ("d2q9", (1, 31, 2), 1), ("d2q9", (1, 33, 5), 0),
                                                ("d2q9", (1, 128, 3), 0), ("d2q9", (1, 257, 3), 1),
                                                ("d3q27", (17, 61, 4), 0), ("d3q27", (1, 2050, 2), 1)])
@pytest.mark.parametrize("nan_at", [None, 0])
def test_nusselt_numbers_are_those_of_the_profile(lattice, shape, face, nan_at):
    """Mean, extrema and their first places against the profile, for faces of one thread up to several
    blocks; a node that is NaN counts for neither extremum and makes the mean NaN.  The mean's sum of
    n FP64 terms in another order: n 2^-52 of the largest."""
    nz, ny, nx = shape
    lat = L.Lattice(lattice, nx, ny, nz, Ra=1e4, precision="fp64")
    f, g = lat.get_populations()
    g = synth.perturbed(g, 7, 0.1)
    if nan_at is not None:
        g[0, 0, 0, nx - 1 if face else 0] = np.nan     # the rest link of the face's first node
    lat.set_populations(f, g)
    prof = lat.nusselt_profile(face).cpu().numpy()
    mean, mx, mn, jmx, jmn = lat.nusselt(face)
    lat.close()
    assert prof.size == ny * nz
    if nan_at is None:
        assert mean == pytest.approx(prof.mean(), abs=prof.size * 2.0 ** -52 * np.abs(prof).max())
    else:
        assert np.isnan(mean) and np.isnan(prof[0])
        if prof.size == 1:
            assert mx == -np.inf and mn == np.inf
            return
    assert (mx, mn) == (np.nanmax(prof), np.nanmin(prof))
    assert (jmx, jmn) == (int(np.nanargmax(prof)), int(np.nanargmin(prof)))


def test_wall_profile_into_unaligned_device_memory():
    """The profile's destination may start at any byte of device memory."""
    lat = L.Lattice("d2q9", 24, 37, Ra=1e4, precision="fp32")
    lat.step(3)
    want = lat.nusselt_profile(0)
    buf = torch.zeros(8 * 37 + 8, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    L.lbm_nusselt_profile(lat.h, 0, buf.data_ptr() + 4, 37, 1)
    got = np.frombuffer(buf.cpu().numpy()[4:4 + 8 * 37].tobytes(), dtype=np.float64)
    lat.close()
    np.testing.assert_array_equal(got, torch.as_tensor(want).cpu().numpy().reshape(-1))


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16s"])
@pytest.mark.parametrize("kind,shape", [("rb", (1, 5, 1)), ("cavity", (1, 300, 3)), ("rb", (1, 7, 31)), ("cavity", (1, 9, 33)),
                                        ("cavity", (1, 4, 56)), ("rb", (1, 5, 55)), ("cavity", (1, 3, 160)), ("rb", (1, 2, 129)),
                                        ("cavity", (3, 5, 2)), ("mixed3d", (4, 3, 21)), ("mixed3d", (2, 7, 22)),
                                        ("cavity", (3, 4, 33)), ("mixed3d", (3, 2, 64)), ("periodic", (3, 5, 65))])
def test_fields_of_narrow_and_ragged_rows(kind, shape, precision):
    """Both ways of dealing nodes to threads, about the row lengths where they change over (a third, an
    eighth or a 32nd of a row's lanes idle) and where warps span several rows, against the oracle's fields.  FP64: a
    few dozen operations on numbers of order one; FP32: its 27 (15) terms' rounding, 2^-24 each; FP16:
    2^-11 of each of the stored deviations, which add up to 0.05 here, over a density of 0.9 or more."""
    dim = 2 if shape[0] == 1 and kind != "mixed3d" else 3
    nz, ny, nx = shape
    gpu, ora = make_pair(dim, nx, ny, nz, kind=kind, precision=precision)
    randomize(gpu, ora, seed=9, scale=0.05)
    got, want = gpu.fields(), ora.fields()
    gpu.close()
    tol = {"fp64": 1e-14, "fp32": 28 * 2.0 ** -24, "fp16s": 0.1 * 2.0 ** -11}[precision]
    for k in ("rho", "ux", "uy", "uz", "T"):
        np.testing.assert_allclose(got[k].cpu().numpy(), want[k], rtol=0, atol=tol, err_msg=k)

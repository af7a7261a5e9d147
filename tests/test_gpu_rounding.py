"""Rounding of single operations and updates, where whole runs would hide it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

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

"""The reduced steps of the default rates against the oracle and against the general collision.

The rates lbm_create sets, with option A and gravity along y (2D) or z (3D), take a step of their own.
FP64 is held to the bars of the other parity tests (1e-14 after one step, 1e-12 after 100 from
perturbed states: both sides compute in FP64 from identical inputs); every storage form is also
compared with the general collision, which one rate moved by 1e-12 selects: a moment's update then
changes by 1e-12 of itself, so the two differ by the rounding of the register type alone.
"""
import numpy as np
import pytest

from oracle import oracle as O
from tests import synth
from tests.test_gpu_parity import make_pair, pop_error, randomize, walls_pair

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_09041_gb300 import lbm as L  # noqa: E402

BOXES = [(2, "cavity", (1, 33, 70)), (2, "rb", (1, 19, 131)), (2, "periodic", (1, 64, 32)),
         (2, "cavity", (1, 3, 2)), (2, "rb", (1, 1, 5)),
         (3, "cavity", (13, 21, 37)), (3, "mixed3d", (9, 10, 70)), (3, "periodic", (5, 6, 33)),
         (3, "mixed3d", (2, 3, 1))]


@pytest.mark.parametrize("gbeta", [None, 3e-3])
@pytest.mark.parametrize("dim,kind,shape", BOXES)
def test_fp64_matches_oracle_at_default_rates(dim, kind, shape, gbeta):
    """gbeta 3e-3 (the box's own is about 1e-5) makes every force term of the sources count."""
    nz, ny, nx = shape
    gpu, ora = make_pair(dim, nx, ny, nz, kind=kind)
    if gbeta is not None:
        gpu.set_param("gbeta", gbeta)
        wo = walls_pair(kind, dim)[1]
        ora = O.Oracle(dim, nx, ny, nz, bc=wo, om_f=ora.om_f, om_g=ora.om_g, gbeta=gbeta)
    randomize(gpu, ora, seed=5, scale=0.1 if dim == 2 else 0.05)
    gpu.step(1)
    ora.step(1)
    assert pop_error(gpu, ora) <= 1e-14
    gpu.step(99)
    ora.step(99)
    gpu.sync()
    assert pop_error(gpu, ora) <= 1e-12


# one step from the same state: values of order 0.1 pass through a few hundred operations
STEP_TOL = {"fp64": 1e-15, "fp32": 2e-7}


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16s"])
@pytest.mark.parametrize("dim,kind,shape", BOXES)
def test_reduced_step_equals_general_collision(dim, kind, shape, precision):
    """FP16 storage rounds to nearest here, so each value differs by at most one step of its
    format (2^-10 of its scaled deviation, at most 2^-10 of the largest)."""
    nz, ny, nx = shape
    lat = "d2q9" if dim == 2 else "d3q27"
    out = []
    for om0 in (1.0, 1.0 + 1e-12):
        gpu = L.Lattice(lat, nx, ny, nz, Ra=1e4, walls=walls_pair(kind, dim)[0], precision=precision)
        inf = gpu.info()
        om_f = np.array(inf.om_f[:inf.q_f])
        om_f[0] = om0
        gpu.set_omegas(om_f, np.array(inf.om_g[:inf.q_g]))
        gpu.set_param("gbeta", 3e-3)
        if precision == "fp16s":
            gpu.set_param("fp16_stochastic", 0)
        f, g = gpu.get_populations()
        gpu.set_populations(synth.perturbed(f, 3, 0.05), synth.perturbed(g, 4, 0.05))
        start = gpu.get_populations()
        gpu.step(1)
        gpu.sync()
        out.append(gpu.get_populations())
        gpu.close()
    for k in (0, 1):
        diff = np.abs(out[0][k] - out[1][k]).max()
        if precision == "fp16s":
            rest = L.Lattice(lat, nx, ny, nz, Ra=1e4, walls=walls_pair(kind, dim)[0], precision="fp64")
            dev = np.abs(out[1][k] - rest.get_populations()[k]).max()
            rest.close()
            assert diff <= 2.0 ** -10 * dev
        else:
            assert diff <= STEP_TOL[precision]
    assert np.abs(out[0][0] - start[0]).max() > 0


@pytest.mark.parametrize("kind,shape,stochastic", [("cavity", (150, 160, 254), 1), ("mixed3d", (97, 251, 258), 0),
                                                   ("periodic", (61, 1541, 64), 1), ("cavity", (2, 3, 1000002), 1),
                                                   ("mixed3d", (1000, 3001, 2), 1)])
def test_fp16s_node_pairs_equal_single_nodes(kind, shape, stochastic):
    """Boxes of six million nodes and more with an even nx update two nodes per thread; rows3d = 1 selects
    the one-node kernel.  Bitwise equal, walls and periodic ends included, after steps that move
    values through each of them; an odd number of steps, so that both walking directions run."""
    nz, ny, nx = shape
    states = []
    for rows in (0, 1):
        gpu = L.Lattice("d3q27", nx, ny, nz, Ra=1e4, walls=walls_pair(kind, 3, seed=5, perturb=0.05)[0],
                        precision="fp16s")
        gpu.set_param("fp16_stochastic", stochastic)
        gpu.set_param("gbeta", 3e-3)
        if rows:
            gpu.set_param("rows3d", rows)
        gpu.step(5)
        gpu.sync()
        states.append(gpu.get_state()[64:])
        gpu.close()
    assert np.array_equal(states[0], states[1])


@pytest.mark.parametrize("kind,shape", [("cavity", (1, 64, 64)), ("rb", (1, 33, 70)), ("periodic", (1, 5, 31)),
                                        ("cavity", (1, 3, 2)), ("rb", (1, 1, 5)), ("cavity", (1, 149, 96)),
                                        ("rb", (1, 448, 32)), ("rb", (1, 449, 32))])
def test_fp64_split_step_equals_the_one_warp_step(kind, shape):
    """Small FP64 boxes run the two lattices of a node on two warps; a chosen block_x selects the
    one-warp kernel.  Bitwise equal up to and just above the size where the rule changes over."""
    nz, ny, nx = shape
    states = []
    for block in (0, 32):
        gpu = L.Lattice("d2q9", nx, ny, Ra=1e4, walls=walls_pair(kind, 2)[0], precision="fp64")
        gpu.set_param("gbeta", 3e-3)
        if block:
            gpu.set_param("block_x", block)
        f, g = gpu.get_populations()
        gpu.set_populations(synth.perturbed(f, 3, 0.05), synth.perturbed(g, 4, 0.05))
        gpu.step(40)
        gpu.sync()
        states.append(gpu.get_state()[64:])
        gpu.close()
    assert np.array_equal(states[0], states[1])


@pytest.mark.parametrize("kind,shape,stochastic", [("cavity", (1, 601, 500), 1), ("rb", (1, 512, 1024), 0),
                                                   ("periodic", (1, 131070, 4), 1), ("rb", (1, 3, 131074), 1)])
def test_fp16s_node_pairs_equal_single_nodes_2d(kind, shape, stochastic):
    """Boxes of 300,000 nodes and more with an even nx update two nodes per thread; a chosen block_x
    selects the one-node kernel.  Bitwise equal; an odd number of steps, so that both walking
    directions run."""
    nz, ny, nx = shape
    states = []
    for block in (0, 64):
        gpu = L.Lattice("d2q9", nx, ny, Ra=1e4, walls=walls_pair(kind, 2, seed=5, perturb=0.05)[0], precision="fp16s")
        gpu.set_param("fp16_stochastic", stochastic)
        gpu.set_param("gbeta", 3e-3)
        if block:
            gpu.set_param("block_x", block)
        gpu.step(5)
        gpu.sync()
        states.append(gpu.get_state()[64:])
        gpu.close()
    assert np.array_equal(states[0], states[1])


@pytest.mark.parametrize("precision,shape", [("fp64", (2, 65537, 3)), ("fp32", (2, 65537, 3)), ("fp16s", (2, 65537, 3)),
                                             ("fp32", (1, 131070, 4)), ("fp16s", (24, 65537, 4))])
def test_3d_boxes_taller_than_the_launch_grid(precision, shape):
    """More than 65535 rows: the default blocks hold two.  Populations equal those of chosen 32 x 8
    blocks bit by bit.  The read-out covers every row too: the collision conserves the temperature, so
    the field is the sum of the energy populations after one more step (FP64 to 1e-13; FP32 to 1e-5, 15
    populations' rounding)."""
    nz, ny, nx = shape
    states = []
    for block in (0, 8):
        gpu = L.Lattice("d3q27", nx, ny, nz, Ra=1e4, walls=walls_pair("mixed3d", 3, seed=5, perturb=0.05)[0],
                        precision=precision)
        if block:
            gpu.set_param("block_x", 32)
            gpu.set_param("block_y", block)
        gpu.step(3)
        gpu.sync()
        states.append(gpu.get_state()[64:])
        if not block and precision != "fp16s":
            T = gpu.fields()["T"].cpu().numpy()
            gpu.step(1)
            _, g = gpu.get_populations()
            np.testing.assert_allclose(g.sum(axis=0), T, rtol=0, atol=1e-13 if precision == "fp64" else 1e-5)
        gpu.close()
    assert np.array_equal(states[0], states[1])

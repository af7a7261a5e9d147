"""FP16 storage, two nodes per thread, against one node per thread from states that differ at every node:
every wrap, wall and row end then carries values of its own, bit by bit."""
import pytest

from tests.test_gpu_parity import walls_pair

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_09041_gb300 import lbm as L  # noqa: E402


# 2D: from 300,000 nodes, row lengths that fill one, two, three and four warps of pairs, the tallest launch grid
# in both block shapes, and beyond L2 a partly filled row.  3D: from six million.
@pytest.mark.parametrize("lattice,kind,shape,stochastic", [
    ("d2q9", "periodic", (1, 4700, 64), 1), ("d2q9", "periodic", (1, 131070, 34), 1), ("d2q9", "periodic", (1, 131070, 98), 0),
    ("d2q9", "cavity", (1, 2401, 126), 1), ("d2q9", "rb", (1, 1600, 190), 1), ("d2q9", "periodic", (1, 1301, 256), 0),
    ("d2q9", "cavity", (1, 15001, 130), 1), ("d2q9", "rb", (1, 6, 131072), 1),
    ("d3q27", "periodic", (61, 1541, 64), 1), ("d3q27", "periodic", (40, 600, 258), 0), ("d3q27", "cavity", (150, 160, 254), 1),
    ("d3q27", "mixed3d", (97, 251, 258), 1), ("d3q27", "periodic", (2, 24001, 126), 1)])
def test_node_pairs_equal_single_nodes_from_any_state(lattice, kind, shape, stochastic):
    nz, ny, nx = shape
    dim = 2 if lattice == "d2q9" else 3
    states = []
    for single in (0, 1):
        lat = L.Lattice(lattice, nx, ny, nz, Ra=1e4, walls=walls_pair(kind, dim)[0], precision="fp16s")
        lat.set_param("fp16_stochastic", stochastic)
        lat.set_param("gbeta", 3e-3)
        if single:
            lat.set_param("block_x" if dim == 2 else "rows3d", 64 if dim == 2 else 1)
        gen = torch.Generator(device="cuda").manual_seed(17)
        start = [p * (1 + 0.05 * (2 * torch.rand(p.shape, generator=gen, device="cuda", dtype=torch.float64) - 1))
                 for p in lat.get_populations(device=True)]
        lat.set_populations(*start)
        start = lat.get_populations(device=True)
        lat.step(5)          # odd, so that both walking directions run
        lat.sync()
        states.append([start, lat.get_populations(device=True)])
        lat.close()
    for k in (0, 1):
        assert torch.equal(states[0][0][k], states[1][0][k])
        assert torch.equal(states[0][1][k], states[1][1][k])
        changed = states[0][1][k] != states[0][0][k]
        # every face and the interior moved on
        for face in (changed[:, 0], changed[:, -1], changed[:, :, 0], changed[:, :, -1], changed[..., 0], changed[..., -1],
                     changed):
            assert face.double().mean() > 0.9
